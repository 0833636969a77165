// Dynamics detection (ReFusion Sec. III-C) on sm_103a.
//
//   k_seeds      r_i = V_SDF(T x_i)^2 (the residual of Eq. 2, V_SDF truncated to
//                [-tau, tau]) and the raw mask r_i > t = gamma tau^2 (Eq. 5), a
//                warp per 32 pixels of a row, written as bits.  The
//                decision is exact: the FP32 evaluation carries an error bound;
//                when the lattice cell or the comparison is within it, the pixel
//                is re-evaluated in float pairs with a far smaller bound, and
//                within that one in FP64 with a fixed operation order and no
//                contraction (__d*_rn), the order the FP64 oracle uses.  The
//                warps also write the pixels' join conditions of Alg. 1, as bits.
//   k_mask_fill  the rest, in one cooperative launch: M_R = 3x3 erosion of the raw
//                mask (outside the image = 0); the closure of Alg. 1, in which n
//                joins from p when |D(p) - D(n)| < theta D(p) (4-neighbours, raw
//                integer depth, theta in ppm); the final mask = 3x3 dilation of
//                M_D.  The closure is the set reachable from M_R, independent of
//                visiting order, so it is taken tile by tile until nothing changes:
//                at most max_ff_sweeps sweeps over the image, a grid-wide barrier
//                (bounded) after each.
#include <cmath>
#include <mutex>

#include "rf_volume.hpp"

namespace rf {
namespace {

// FP64 residual in the fixed evaluation order; r < 0 when the lookup is invalid.
template <int ST>
__device__ double residual_fp64(const DevVol& v, const DevFrame& f, const DevParams& p, const double* T, int u, int vv,
                                unsigned raw) {
  const double D = __ddiv_rn((double)raw, p.depth_scale_d);
  const double x = __dmul_rn(__ddiv_rn(__dsub_rn((double)u, f.cxd), f.fxd), D);
  const double y = __dmul_rn(__ddiv_rn(__dsub_rn((double)vv, f.cyd), f.fyd), D);
  const double z = D;
  double q[3];
  int k[3];
  double fr[3];
  for (int i = 0; i < 3; ++i) {
    const double pi = __dadd_rn(
        __dadd_rn(__dadd_rn(__dmul_rn(T[i * 4 + 0], x), __dmul_rn(T[i * 4 + 1], y)), __dmul_rn(T[i * 4 + 2], z)),
        T[i * 4 + 3]);
    q[i] = __ddiv_rn(pi, p.voxel_d);
    if (!(fabs(q[i]) < 1e9)) return -1.0;
    const double fl = floor(q[i]);
    k[i] = (int)fl;
    fr[i] = __dsub_rn(q[i], fl);
  }
  if (abs(k[0]) > 8 * kMaxCoord || abs(k[1]) > 8 * kMaxCoord || abs(k[2]) > 8 * kMaxCoord) return -1.0;
  float F[8];
  if (!corners_of<ST>(v, p, k[0], k[1], k[2], F)) return -1.0;
  const double c00 = lerp_rn(F[0], F[1], fr[0]), c10 = lerp_rn(F[2], F[3], fr[0]);
  const double c01 = lerp_rn(F[4], F[5], fr[0]), c11 = lerp_rn(F[6], F[7], fr[0]);
  const double c0 = lerp_rn(c00, c10, fr[1]), c1 = lerp_rn(c01, c11, fr[1]);
  const double V = fmin(fmax(lerp_rn(c0, c1, fr[2]), -p.tau_d), p.tau_d);  // truncated at tau
  return __dmul_rn(V, V);
}

// Seed decision from the cell's corners and the position in it, known within
// eps_q: 0 or 1, or 2 when the comparison lies within the error bound.
__device__ __forceinline__ int seed_of(const DevParams& p, const float F[8], const float fr[3], float eps_q) {
  const float t = p.gamma_tau2_f;
  const float c00 = F[0] * (1.0f - fr[0]) + F[1] * fr[0], c10 = F[2] * (1.0f - fr[0]) + F[3] * fr[0];
  const float c01 = F[4] * (1.0f - fr[0]) + F[5] * fr[0], c11 = F[6] * (1.0f - fr[0]) + F[7] * fr[0];
  const float c0 = c00 * (1.0f - fr[1]) + c10 * fr[1], c1 = c01 * (1.0f - fr[1]) + c11 * fr[1];
  const float V = fminf(fmaxf(c0 * (1.0f - fr[2]) + c1 * fr[2], -p.tau), p.tau);
  float fmn = F[0], fmx = F[0], fab = fabsf(F[0]);
#pragma unroll
  for (int n = 1; n < 8; ++n) {
    fmn = fminf(fmn, F[n]);
    fmx = fmaxf(fmx, F[n]);
    fab = fmaxf(fab, fabsf(F[n]));
  }
  // + the gap between the float and double truncation bounds (<= 2^-24 tau)
  const float dV = 3.0f * (fmx - fmn) * eps_q + fab * 1.9073486328125e-06f + p.tau * 5.9604645e-08f;
  const float r = V * V;
  const float dr = 2.0f * fabsf(V) * dV + dV * dV + r * 2.384185791015625e-07f;  // 2^-22
  if (fabsf(r - t) <= 2.0f * dr + t * 2.384185791015625e-07f) return 2;
  return r > t ? 1 : 0;
}

// Seed decision of one valid pixel in FP32 with an error bound: 0 or 1, or
// 2 when the lattice cell or the comparison lies within the bound (the pixel
// is then decided in float pairs or FP64).  Rf: the pose as floats (R row-major, then t).
template <int ST>
__device__ __forceinline__ int seed_fp32(const DevVol& v, const DevFrame& f, const DevParams& p, const float* Rf, int u,
                                         int vv, unsigned raw, unsigned long long cached) {
  const float D = (float)raw * p.inv_depth_scale;
  const float x = ((float)u - f.cx) * f.ifx * D, y = ((float)vv - f.cy) * f.ify * D;
  float q[3], fr[3];
  int k[3];
  const float mag_in = (fabsf(x) + fabsf(y) + fabsf(D) + fabsf(Rf[9]) + fabsf(Rf[10]) + fabsf(Rf[11])) * p.inv_voxel;
  float qmax = 0.0f;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float pi = Rf[i * 3] * x + Rf[i * 3 + 1] * y + Rf[i * 3 + 2] * D + Rf[9 + i];
    q[i] = pi * p.inv_voxel;
    qmax = fmaxf(qmax, fabsf(q[i]));
  }
  // bound on |q32 - q64| with an 8x margin (see the error budget in the design notes)
  const float eps_q = (mag_in + qmax) * 3.814697265625e-06f;  // 2^-18
  if (!(qmax < 8.0f * kMaxCoord - 2.0f)) return 2;
  bool ambiguous = false;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float fl = floorf(q[i]);
    k[i] = (int)fl;
    fr[i] = q[i] - fl;
    if (fr[i] < eps_q || fr[i] > 1.0f - eps_q) ambiguous = true;
  }
  if (ambiguous) return 2;
  float F[8];
  // an unambiguous cell with a missing corner is invalid in FP64 too: no seed
  if (!corners_cached<ST>(v, p, k[0], k[1], k[2], cached, F)) return 0;
  return seed_of(p, F, fr, eps_q);
}

// The same in float pairs.
template <int ST>
__device__ __forceinline__ int seed_ff(const DevVol& v, const DevFrame& f, const DevParams& p, const FF* T, int u, int vv,
                                       unsigned raw) {
  const FF D = ff_mul(FF{(float)raw, 0.0f}, FF{p.inv_depth_scale, p.inv_depth_scale_lo});
  int k[3];
  float fr[3], F[8];
  if (!cell_ff(f, p, T, u, vv, D, k, fr)) return 2;
  if (!corners_of<ST>(v, p, k[0], k[1], k[2], F)) return 0;
  return seed_of(p, F, fr, kFrErrFF);
}

__device__ __forceinline__ bool may_join(unsigned from, unsigned to, long long theta_ppm) {
  const unsigned diff = from > to ? from - to : to - from;
  return (long long)((unsigned long long)diff * 1000000u) < theta_ppm * (long long)from;
}

// Words of one tile of 32 x 32 pixels, row r of each plane at word 32 plane +
// r: raw mask, joins from the left, from the right (bits reversed), from
// above and from below, the flood fill's set M; then M's border: top row,
// bottom row, left column, right column.
constexpr int kSeedsPlane = 0, kRightPlane = 32, kLeftPlane = 64, kDownPlane = 96, kUpPlane = 128, kMPlane = 160,
              kBorder = 192;
static_assert(kBorder + 4 == kFillTileWords, "tile layout");

// Seeds and join conditions of the kSeedThreads / 32 * kSeedPx row words (32
// pixels of a row, the first one's column a multiple of 32) of CTA `block`.
// Every thread first loads its pixels' depths and cache entries, then decides
// them in FP32; the ambiguous ones (~2 %, almost all for their lattice cell)
// are queued in shared memory and decided in float pairs afterwards, side by
// side by consecutive threads, and what that leaves open (one in thousands of
// them) in FP64, whose chain alone took half the kernel's time.
// The join conditions of Alg. 1 are decided here, where every SM has pixels and
// the issue slots are idle (the lookups' latency bounds the kernel), and not in
// the flood fill, which runs on few SMs (there they took 13 us of 640x480).
// pxcache: the registration's per-pixel block cache, read only, to skip hash
// probes.
constexpr int kSeedThreads = 256;
constexpr int kSeedPx = 4;
constexpr int kSeedWords = kSeedThreads / 32 * kSeedPx;

__host__ __device__ constexpr int row_words(int W) { return (W + 31) / 32; }
__host__ __device__ constexpr int seed_blocks(int H, int W) { return (H * row_words(W) + kSeedWords - 1) / kSeedWords; }

template <int ST>
__device__ __forceinline__ void seeds_body(const DevVol& v, const DevFrame& f, const DevParams& p,
                                           const double* __restrict__ T, unsigned* __restrict__ tiles,
                                           unsigned* guard_count, const unsigned long long* __restrict__ pxcache,
                                           int block) {
  // pose converted once per CTA (conversions use the FP64 pipe)
  __shared__ float sR[12];
  __shared__ unsigned short s_queue[kSeedWords * 32];
  __shared__ unsigned s_words[kSeedWords];
  __shared__ int s_n, s_open, s_last[kSeedThreads];
  __shared__ FF s_T[12];
  if (threadIdx.x < 12) {
    const int i = threadIdx.x < 9 ? threadIdx.x / 3 : threadIdx.x - 9;
    const int j = threadIdx.x < 9 ? threadIdx.x % 3 : 3;
    sR[threadIdx.x] = (float)T[i * 4 + j];
  }
  if (threadIdx.x == 13) s_n = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rw = row_words(f.W), nwords = f.H * rw;
  auto word_of = [&](int local) { return block * kSeedWords + local; };  // local: 0 .. kSeedWords - 1
  auto tile_word = [&](int w) {  // the place of row word w in its tile's planes
    const int row = w / rw;
    return tiles + (size_t)((row >> 5) * rw + (w - row * rw)) * kFillTileWords + (row & 31);
  };
  unsigned raw[kSeedPx], above[kSeedPx], below[kSeedPx], side[kSeedPx];
  unsigned long long cached[kSeedPx];
  int us[kSeedPx], vs[kSeedPx];
#pragma unroll
  for (int j = 0; j < kSeedPx; ++j) {
    const int w = word_of(j * (kSeedThreads / 32) + warp), row = w / rw;
    const int u = (w - row * rw) * 32 + lane, idx = row * f.W + u;
    const bool in = w < nwords && u < f.W;
    us[j] = u;
    vs[j] = row;
    raw[j] = in ? __ldg(f.depth + idx) : 0u;
    cached[j] = in ? __ldg(pxcache + idx) : kEmpty;
    above[j] = in && row > 0 ? __ldg(f.depth + idx - f.W) : 0u;
    below[j] = in && row + 1 < f.H ? __ldg(f.depth + idx + f.W) : 0u;
    side[j] = in && lane == 0 && u > 0 ? __ldg(f.depth + idx - 1)
              : in && lane == 31 && u + 1 < f.W ? __ldg(f.depth + idx + 1)
                                                : 0u;
  }
#pragma unroll 1
  for (int j = 0; j < kSeedPx; ++j) {
    const int local = j * (kSeedThreads / 32) + warp, w = word_of(local);
    if (w >= nwords) break;
    const unsigned rj = j == 0 ? raw[0] : (j == 1 ? raw[1] : (j == 2 ? raw[2] : raw[3]));
    const unsigned aj = j == 0 ? above[0] : (j == 1 ? above[1] : (j == 2 ? above[2] : above[3]));
    const unsigned bj = j == 0 ? below[0] : (j == 1 ? below[1] : (j == 2 ? below[2] : below[3]));
    const unsigned sj = j == 0 ? side[0] : (j == 1 ? side[1] : (j == 2 ? side[2] : side[3]));
    const unsigned long long cj = j == 0 ? cached[0] : (j == 1 ? cached[1] : (j == 2 ? cached[2] : cached[3]));
    const int u = j == 0 ? us[0] : (j == 1 ? us[1] : (j == 2 ? us[2] : us[3]));
    const int vv = j == 0 ? vs[0] : (j == 1 ? vs[1] : (j == 2 ? vs[2] : vs[3]));
    int seed = 0;
    if (pixel_valid(p, rj)) seed = seed_fp32<ST>(v, f, p, sR, u, vv, rj, cj);  // (raw is 0 outside the image)
    if (seed == 2) s_queue[atomicAdd(&s_n, 1)] = (unsigned short)(local * 32 + lane);
    __syncwarp();
    const unsigned seeds = __ballot_sync(0xffffffffu, seed == 1);
    // join conditions (a depth of 0, also outside the image, joins nothing)
    const unsigned dl = __shfl_up_sync(0xffffffffu, rj, 1), dr = __shfl_down_sync(0xffffffffu, rj, 1);
    const unsigned jr = __ballot_sync(0xffffffffu, may_join(lane == 0 ? sj : dl, rj, p.theta_ppm));
    const unsigned jl = __ballot_sync(0xffffffffu, may_join(lane == 31 ? sj : dr, rj, p.theta_ppm));
    const unsigned jd = __ballot_sync(0xffffffffu, may_join(aj, rj, p.theta_ppm));
    const unsigned ju = __ballot_sync(0xffffffffu, may_join(bj, rj, p.theta_ppm));
    if (lane == 0) s_words[local] = seeds;
    if (lane < 4) {
      const unsigned x = lane == 0 ? jr : (lane == 1 ? __brev(jl) : (lane == 2 ? jd : ju));
      tile_word(w)[kRightPlane + 32 * lane] = x;
    }
  }
  if (threadIdx.x < 12) {  // the pose in float pairs
    const double t = T[threadIdx.x];
    const float h = (float)t;
    s_T[threadIdx.x] = FF{h, (float)(t - (double)h)};
  }
  __syncthreads();
  const int n = s_n;
  // the ambiguous pixels in float pairs, then those that remain so in FP64
  auto pixel_of = [&](int q, int& u, int& row) {
    const int w = word_of(q >> 5);
    row = w / rw;
    u = (w - row * rw) * 32 + (q & 31);
  };
  for (int i0 = 0; i0 < n; i0 += kSeedThreads) {
    if (threadIdx.x == 0) s_open = 0;
    __syncthreads();
    const int i = i0 + (int)threadIdx.x;
    if (i < n) {
      const int q = s_queue[i];
      int u, row;
      pixel_of(q, u, row);
      const int seed = seed_ff<ST>(v, f, p, s_T, u, row, __ldg(f.depth + row * f.W + u));
      if (seed == 1) atomicOr(&s_words[q >> 5], 1u << (q & 31));
      if (seed == 2) s_last[atomicAdd(&s_open, 1)] = q;
    }
    __syncthreads();
    if ((int)threadIdx.x < s_open) {
      const int q = s_last[threadIdx.x];
      int u, row;
      pixel_of(q, u, row);
      const double r64 = residual_fp64<ST>(v, f, p, T, u, row, __ldg(f.depth + row * f.W + u));
      if (r64 >= 0.0 && r64 > __dmul_rn(__dmul_rn(p.gamma_d, p.tau_d), p.tau_d))
        atomicOr(&s_words[q >> 5], 1u << (q & 31));
    }
    __syncthreads();  // s_open is reset next
  }
  if (threadIdx.x == 0 && n > 0 && guard_count) atomicAdd(guard_count, (unsigned)n);
  __syncthreads();
  if (threadIdx.x < kSeedWords && word_of(threadIdx.x) < nwords)
    tile_word(word_of(threadIdx.x))[kSeedsPlane] = s_words[threadIdx.x];
}

template <int ST>
__global__ void __launch_bounds__(kSeedThreads) k_seeds(DevVol v, DevFrame f, DevParams p,
                                                        const double* __restrict__ T, unsigned* __restrict__ tiles,
                                                        unsigned* guard_count,
                                                        const unsigned long long* __restrict__ pxcache) {
  seeds_body<ST>(v, f, p, T, tiles, guard_count, pxcache, blockIdx.x);
}

// grid (x, n streams): the seeds of every tracked stream of a batch.
template <int ST>
__global__ void __launch_bounds__(kSeedThreads) k_seeds_batch(const MaskDesc* __restrict__ descs) {
  const MaskDesc& d = descs[blockIdx.y];
  if (gated_off(d.f.gate, kModeTrack) || (int)blockIdx.x >= seed_blocks(d.f.H, d.f.W)) return;
  seeds_body<ST>(d.v, d.f, d.p, d.T, d.tiles, d.guard, d.pxcache, blockIdx.x);
}

// ---------------------------------------------------------------------------
// Erosion, flood fill and dilation.  A warp holds a tile of 32 x 32 pixels as
// bits, row r on lane r: the set M and four planes of join conditions (bit c
// of row r: the pixel may join from its left / right / upper / lower
// neighbour).  Within the tile a row fills to either side with one addition
// (the carry runs through the joinable pixels) and the columns in five shuffle
// steps each way, so a tile settles in a few hundred cycles, where a pixel per
// thread and step took up to 512 CTA barriers.  The 4 x 4 tiles of a CTA
// exchange their border rows and columns through shared memory until none
// changes, then CTAs exchange theirs through global memory, a grid barrier per
// sweep: an object of a few hundred pixels takes three or four sweeps.  Bound
// by latency: barriers, and the chain of tiles an object extends over.
// 640x480 with a moving object: erosion, fill and dilation 50 us before (three
// kernels, 600 tiles of 32 x 16 in ~12 sweeps).
// ---------------------------------------------------------------------------
constexpr int kFillTx = 4, kFillTy = 4;  // tiles of a CTA's region
constexpr int kFillThreads = 32 * kFillTx * kFillTy;
// One tile in a warp's registers.
struct Tile {
  unsigned m;               // M
  unsigned right, left_r;   // joins from the left neighbour, and (bits reversed) from the right one
  unsigned down, up;        // joins from above and from below
};

// Bits of the row words that a fill towards higher bits reaches: `p` marks the
// pixels that may join from the next lower bit.  Adding the first joining
// pixels to p clears the run of ones above each of them.
__device__ __forceinline__ unsigned fill_up_bits(unsigned m, unsigned p) {
  const unsigned s = p & (m << 1), sum = p + s;
  return m | s | (p & ~sum);
}

// Closure within the tile.
__device__ __forceinline__ unsigned settle(Tile t, int lane) {
  unsigned pd[5], pu[5];  // rows 1, 2, 4, 8, 16 above / below reach this one
  pd[0] = lane == 0 ? 0u : t.down;
  pu[0] = lane == 31 ? 0u : t.up;
#pragma unroll
  for (int k = 0; k < 4; ++k) {  // (a lane without a row that far away gets its own value: 0 there)
    pd[k + 1] = pd[k] & __shfl_up_sync(0xffffffffu, pd[k], 1 << k);
    pu[k + 1] = pu[k] & __shfl_down_sync(0xffffffffu, pu[k], 1 << k);
  }
  unsigned m = t.m, old;
  do {
    old = m;
    m = fill_up_bits(m, t.right);
    m = __brev(fill_up_bits(__brev(m), t.left_r));
#pragma unroll
    for (int k = 0; k < 5; ++k) m |= pd[k] & __shfl_up_sync(0xffffffffu, m, 1 << k);
#pragma unroll
    for (int k = 0; k < 5; ++k) m |= pu[k] & __shfl_down_sync(0xffffffffu, m, 1 << k);
  } while (__any_sync(0xffffffffu, m != old));  // at most 1,024 times: each adds a pixel
  return m;
}

// M_R, the 3x3 erosion of the raw mask, of tile (tx, ty); zero outside the
// image.  All words are loaded before any is used.
__device__ __forceinline__ unsigned erode_tile(const unsigned* __restrict__ tiles, int tiles_x, int H, int tx, int ty,
                                               int lane) {
  // row words of the tile and its left and right neighbour, of row y of the image
  auto word = [&](int x, int y) {
    return x >= 0 && x < tiles_x && y >= 0 && y < H
               ? __ldcg(tiles + (size_t)((y >> 5) * tiles_x + x) * kFillTileWords + kSeedsPlane + (y & 31))
               : 0u;
  };
  const int y = ty * 32 + lane, ya = ty * 32 - 1, yb = ty * 32 + 32;
  const unsigned w = word(tx, y), l = word(tx - 1, y), r = word(tx + 1, y);
  const unsigned aw = word(tx, ya), al = word(tx - 1, ya), ar = word(tx + 1, ya);
  const unsigned bw = word(tx, yb), bl = word(tx - 1, yb), br = word(tx + 1, yb);
  auto narrow = [](unsigned c, unsigned left, unsigned right) {
    return c & ((c << 1) | (left >> 31)) & ((c >> 1) | (right << 31));
  };
  const unsigned h = narrow(w, l, r), above = narrow(aw, al, ar), below = narrow(bw, bl, br);
  const unsigned hu = __shfl_up_sync(0xffffffffu, h, 1), hd = __shfl_down_sync(0xffffffffu, h, 1);
  return h & (lane == 0 ? above : hu) & (lane == 31 ? below : hd);
}

// Border of M: top row, bottom row, left column, right column (on every lane).
__device__ __forceinline__ uint4 border_of(unsigned m) {
  return make_uint4(__shfl_sync(0xffffffffu, m, 0), __shfl_sync(0xffffffffu, m, 31),
                    __ballot_sync(0xffffffffu, m & 1u), __ballot_sync(0xffffffffu, m >> 31));
}

// ff words: [1] barrier count, [2] barrier generation, [3 + s % 3] changed in
// sweep s, [6] M_R is not empty (all zero at the start; [0] is the seeds' guard
// count).  Run by a group of G CTAs, this one being number lb of the group.
__device__ void mask_fill_body(const FillDesc& d, int lb, int G) {
  __shared__ uint4 sb[2][kFillTx * kFillTy];  // the tiles' borders, by parity of the exchange
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wx = warp % kFillTx, wy = warp / kFillTx;
  const int H = d.H, W = d.W;
  const int tiles_x = (W + 31) / 32, tiles_y = (H + 31) / 32;
  const int regs_x = (tiles_x + kFillTx - 1) / kFillTx;
  const int nreg = regs_x * ((tiles_y + kFillTy - 1) / kFillTy);
  const bool resident = nreg <= G;  // one region per CTA: its tiles stay in registers
  volatile unsigned* changed = d.ff + 3;
  auto tile_at = [&](int tx, int ty) -> int {
    return tx >= 0 && ty >= 0 && tx < tiles_x && ty < tiles_y ? ty * tiles_x + tx : -1;
  };
  auto words = [&](int tile) { return d.tiles + (size_t)tile * kFillTileWords; };
  auto border_word = [&](int tile, int k) { return tile >= 0 ? __ldcg(words(tile) + kBorder + k) : 0u; };
  auto put_border = [&](int tile, const uint4& b) {
    if (lane < 4) __stcg(words(tile) + kBorder + lane, lane == 0 ? b.x : (lane == 1 ? b.y : (lane == 2 ? b.z : b.w)));
  };
  auto load_planes = [&](int tile, int ty, Tile& x) {
    const unsigned* w = words(tile) + lane;
    const bool in = ty * 32 + lane < H;  // (rows below the image were not written)
    x.right = in ? __ldcg(w + kRightPlane) : 0u;
    x.left_r = in ? __ldcg(w + kLeftPlane) : 0u;
    x.down = in ? __ldcg(w + kDownPlane) : 0u;
    x.up = in ? __ldcg(w + kUpPlane) : 0u;
  };
  Tile t = {0u, 0u, 0u, 0u, 0u};
  bool some = false;
  for (int reg = lb; reg < nreg; reg += G) {
    const int tx = reg % regs_x * kFillTx + wx, ty = reg / regs_x * kFillTy + wy, tile = tile_at(tx, ty);
    if (tile < 0) continue;
    t.m = erode_tile(d.tiles, tiles_x, H, tx, ty, lane);
    some = some || t.m != 0u;
    put_border(tile, border_of(t.m));
    if (resident) load_planes(tile, ty, t);
    else __stcg(words(tile) + kMPlane + lane, t.m);
  }
  if (__syncthreads_or(some) && threadIdx.x == 0) atomicExch(d.ff + 6, 1u);
  bool ok = grid_barrier(d.ff + 1, G, d.status, d.spin_limit, d.bar_extra);
  const bool any = ok && *(volatile unsigned*)(d.ff + 6) != 0u;
  bool settled = !any;
  for (int sweep = 0; ok && !settled && sweep < d.max_sweeps; ++sweep) {
    bool grew = false;
    for (int reg = lb; reg < nreg; reg += G) {
      const int tx = reg % regs_x * kFillTx + wx, ty = reg / regs_x * kFillTy + wy, tile = tile_at(tx, ty);
      if (!resident && tile >= 0) {
        t.m = __ldcg(words(tile) + kMPlane + lane);
        load_planes(tile, ty, t);
      }
      if (tile < 0) t = Tile{0u, 0u, 0u, 0u, 0u};
      // facing borders of the tiles around the region (as of the last barrier)
      unsigned top = 0u, bottom = 0u, left = 0u, right = 0u;
      if (tile >= 0) {
        if (wy == 0) top = border_word(tile_at(tx, ty - 1), 1);
        if (wy == kFillTy - 1) bottom = border_word(tile_at(tx, ty + 1), 0);
        if (wx == 0) left = border_word(tile_at(tx - 1, ty), 3);
        if (wx == kFillTx - 1) right = border_word(tile_at(tx + 1, ty), 2);
      }
      const unsigned before = t.m;
      int par = 0;
      uint4 b = border_of(t.m);
      __syncthreads();  // the last region's exchange has been read
      if (lane == 0) sb[0][warp] = b;
      __syncthreads();
      for (;;) {  // at most once per pixel of the region: each round but the last adds one
        const unsigned was = t.m;
        if (wy > 0) top = sb[par][warp - kFillTx].y;
        if (wy < kFillTy - 1) bottom = sb[par][warp + kFillTx].x;
        if (wx > 0) left = sb[par][warp - 1].w;
        if (wx < kFillTx - 1) right = sb[par][warp + 1].z;
        if (lane == 0) t.m |= t.down & top;
        if (lane == 31) t.m |= t.up & bottom;
        t.m |= (left >> lane) & t.right & 1u;
        t.m |= (((right >> lane) & t.left_r) & 1u) << 31;  // (bit 0 of the reversed plane is column 31)
        if (__any_sync(0xffffffffu, t.m != 0u)) t.m = settle(t, lane);
        b = border_of(t.m);
        par ^= 1;
        if (lane == 0) sb[par][warp] = b;
        if (!__syncthreads_or(t.m != was)) break;
      }
      if (tile >= 0 && __any_sync(0xffffffffu, t.m != before)) {
        grew = true;
        put_border(tile, b);
        if (!resident) __stcg(words(tile) + kMPlane + lane, t.m);
      }
    }
    if (__syncthreads_or(grew) && threadIdx.x == 0) atomicExch(d.ff + 3 + sweep % 3, 1u);
    ok = grid_barrier(d.ff + 1, G, d.status, d.spin_limit, d.bar_extra);
    if (!ok) break;
    settled = changed[sweep % 3] == 0u;
    // this sweep's predecessor's flag was read before the barrier; it serves
    // the sweep after next
    if (lb == 0 && threadIdx.x == 0) changed[(sweep + 2) % 3] = 0u;
  }
  if (ok && !settled && lb == 0 && threadIdx.x == 0) atomicOr(d.status, ST_NOT_CONVERGED);
  // dilation, from the tiles and the facing borders of the eight around each
  // (16-byte stores where every row starts on a 16-byte boundary)
  const bool wide_stores = (W & 15) == 0 && (reinterpret_cast<uintptr_t>(d.mask_out) & 15) == 0;
  for (int reg = lb; reg < nreg; reg += G) {
    const int tx = reg % regs_x * kFillTx + wx, ty = reg / regs_x * kFillTy + wy, tile = tile_at(tx, ty);
    if (tile < 0) continue;
    unsigned out = 0u;
    if (any) {
      if (!resident) t.m = __ldcg(words(tile) + kMPlane + lane);
      const unsigned left = border_word(tile_at(tx - 1, ty), 3), right = border_word(tile_at(tx + 1, ty), 2);
      const unsigned wide = t.m | (t.m << 1) | (t.m >> 1) | ((left >> lane) & 1u) | (((right >> lane) & 1u) << 31);
      auto wide_row = [&](int y, int k) {  // the row next to the tile, widened
        const unsigned w = border_word(tile_at(tx, y), k);
        return w | (w << 1) | (w >> 1) | (border_word(tile_at(tx - 1, y), k) >> 31) |
               (border_word(tile_at(tx + 1, y), k) << 31);
      };
      const unsigned above = wide_row(ty - 1, 1), below = wide_row(ty + 1, 0);
      const unsigned wu = __shfl_up_sync(0xffffffffu, wide, 1), wd = __shfl_down_sync(0xffffffffu, wide, 1);
      out = wide | (lane == 0 ? above : wu) | (lane == 31 ? below : wd);
    }
    const int y = ty * 32 + lane;
    if (wide_stores && tx * 32 + 32 <= W) {
      // each lane its row's 32 bytes: a multiplication spreads four bits over four bytes
      unsigned q[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) q[k] = (((out >> (4 * k)) & 15u) * 0x00204081u) & 0x01010101u;
      if (y < H) {
        uint4* o = reinterpret_cast<uint4*>(d.mask_out + (size_t)y * W + tx * 32);
        o[0] = make_uint4(q[0], q[1], q[2], q[3]);
        o[1] = make_uint4(q[4], q[5], q[6], q[7]);
      }
    } else {
      const int u = tx * 32 + lane;
#pragma unroll 8
      for (int r = 0; r < 32; ++r) {
        const unsigned row = __shfl_sync(0xffffffffu, out, r);
        const int v = ty * 32 + r;
        if (u < W && v < H) d.mask_out[(size_t)v * W + u] = (uint8_t)((row >> lane) & 1u);
      }
    }
  }
}

__global__ void __launch_bounds__(kFillThreads) k_mask_fill(FillDesc d) { mask_fill_body(d, blockIdx.x, gridDim.x); }

// The same for several streams in one cooperative launch: CTA b runs stream
// cta_stream[b] (-1: none) as member b - first[s] of its group (the CTA maps
// of the batched registration).  Groups never wait on each other.
__global__ void __launch_bounds__(kFillThreads) k_mask_fill_batch(const FillDesc* __restrict__ descs,
                                                                  const int* __restrict__ cta_stream,
                                                                  const int* __restrict__ first) {
  const int s = cta_stream[blockIdx.x];
  if (s < 0) return;
  mask_fill_body(descs[s], blockIdx.x - first[s], first[s + 1] - first[s]);
}

}  // namespace

static rf_status launch_seeds(rf_volume* vol, const DevFrame& f, const double* T, unsigned* tiles, unsigned* guard,
                              cudaStream_t st) {
  const int blocks = seed_blocks(f.H, f.W);
  if (vol->p.storage == RF_STORAGE_FP16)
    k_seeds<RF_STORAGE_FP16><<<blocks, kSeedThreads, 0, st>>>(vol->dv, f, vol->dp, T, tiles, guard, vol->d_pxcache);
  else
    k_seeds<RF_STORAGE_FP32><<<blocks, kSeedThreads, 0, st>>>(vol->dv, f, vol->dp, T, tiles, guard, vol->d_pxcache);
  return check_cuda(vol, cudaGetLastError(), "seeds launch");
}

static rf_status launch_coop(rf_volume* vol, const void* fn, int grid, void** args, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kFillThreads);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return check_cuda(vol, cudaLaunchKernelExC(&cfg, fn, args), "flood-fill launch");
}

static rf_status launch_fill(rf_volume* vol, FillDesc d, cudaStream_t st) {
  const int rx = (d.W + 32 * kFillTx - 1) / (32 * kFillTx), ry = (d.H + 32 * kFillTy - 1) / (32 * kFillTy);
  void* args[] = {&d};
  return launch_coop(vol, (const void*)k_mask_fill, rx * ry < vol->ff_grid ? rx * ry : vol->ff_grid, args, st);
}

FillDesc make_fill_desc(rf_volume* vol, const DevFrame& f, uint8_t* mask_out) {
  FillDesc d;
  d.mask_out = mask_out;
  d.tiles = vol->d_tiles;
  d.H = f.H;
  d.W = f.W;
  d.ff = vol->d_ff;
  d.max_sweeps = vol->p.max_ff_sweeps;
  d.status = vol->d_status;
  d.spin_limit = vol->wait_spins;
  d.bar_extra = vol->wait_extra;
  return d;
}

rf_status launch_mask(rf_volume* vol, const DevFrame& f, const double* T, uint8_t* mask_out, cudaStream_t st) {
  rf_status s = check_cuda(vol, cudaMemsetAsync(vol->d_ff, 0, sizeof(unsigned) * kFillWords, st), "mask words reset");
  if (s == RF_OK) s = launch_seeds(vol, f, T, vol->d_tiles, vol->d_guard, st);
  if (s == RF_OK) s = launch_fill(vol, make_fill_desc(vol, f, mask_out), st);
  return s;
}

MaskDesc make_mask_desc(rf_volume* vol, const DevFrame& f, const double* T) {
  MaskDesc d;
  d.v = vol->dv;
  d.f = f;
  d.p = vol->dp;
  d.T = T;
  d.tiles = vol->d_tiles;
  d.guard = vol->d_guard;
  d.pxcache = vol->d_pxcache;
  return d;
}

rf_status launch_seeds_batch(rf_volume* vol, const MaskDesc* descs, int n, int max_blocks, cudaStream_t st) {
  const dim3 grid((unsigned)max_blocks, (unsigned)n);
  if (vol->p.storage == RF_STORAGE_FP16)
    k_seeds_batch<RF_STORAGE_FP16><<<grid, kSeedThreads, 0, st>>>(descs);
  else
    k_seeds_batch<RF_STORAGE_FP32><<<grid, kSeedThreads, 0, st>>>(descs);
  return check_cuda(vol, cudaGetLastError(), "batched seeds launch");
}

rf_status launch_fill_batch(rf_volume* vol, const FillDesc* descs, const int* cta_stream, const int* first,
                            int total_ctas, cudaStream_t st) {
  void* args[] = {(void*)&descs, (void*)&cta_stream, (void*)&first};
  return launch_coop(vol, (const void*)k_mask_fill_batch, total_ctas, args, st);
}

int mask_seed_blocks(int H, int W) { return seed_blocks(H, W); }

int floodfill_max_grid(int device) {
  int per_sm = 1 << 20, sms = 0;
  for (const void* fn : {(const void*)k_mask_fill, (const void*)k_mask_fill_batch}) {
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, kFillThreads, 0);
    per_sm = n < per_sm ? n : per_sm;
  }
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  return per_sm * sms;
}

// ---------------------------------------------------------------------------
// Mask without any allocation: the per-call scratch of rf_compute_mask (the
// flood fill's tiles, barrier words, change flags and the guard counter) lives in one file-scope device array instead of the buffers
// the volume owns.  Every GPU that loads this library holds the array (about
// 0.9 MB) until the process exits.
// ---------------------------------------------------------------------------
constexpr int kNoAllocMaxPixels = 1280 * 720;  // largest frame: 921,600 pixels
constexpr int kNoAllocMaxTiles = 1152;          // of frames that size with sides up to 8,192
constexpr int kNoAllocMaxSweeps = 4096;         // flood-fill sweep bound of this entry point
constexpr size_t kNoAllocWordsOff = sizeof(unsigned) * kNoAllocMaxTiles * kFillTileWords;
constexpr size_t kNoAllocBytes = kNoAllocWordsOff + sizeof(unsigned) * kFillWords;

static __device__ __align__(256) unsigned char g_mask_scratch[kNoAllocBytes];

// Device address of g_mask_scratch, looked up once per device with that
// device current.  In host code the symbol is only a host-side stand-in.
static void* mask_scratch_address(int device, cudaError_t* err) {
  static std::mutex mu;
  static void* addr[64] = {};
  *err = cudaSuccess;
  if (device < 0 || device >= 64) {
    *err = cudaErrorInvalidDevice;
    return nullptr;
  }
  std::lock_guard<std::mutex> lock(mu);
  if (!addr[device]) {
    void* p = nullptr;
    *err = cudaGetSymbolAddress(&p, g_mask_scratch);
    if (*err != cudaSuccess) return nullptr;
    addr[device] = p;
  }
  return addr[device];
}

}  // namespace rf

using namespace rf;

extern "C" rf_status rf_compute_mask_noalloc(rf_volume* vol, const rf_frame* frame, const double* T_dev,
                                             uint8_t* mask_dev, void* stream) {
  if (!vol) return RF_ERR_INVALID_ARG;
  if (!frame_ok(vol, frame)) return set_error(vol, RF_ERR_INVALID_ARG, "invalid frame");
  if (!T_dev || !mask_dev) return set_error(vol, RF_ERR_INVALID_ARG, "NULL pose or mask");
  if ((int64_t)frame->height * frame->width > kNoAllocMaxPixels)
    return set_error(vol, RF_ERR_INVALID_ARG,
                     "rf_compute_mask_noalloc: frame of %d x %d pixels exceeds the static scratch limit of %d pixels",
                     frame->width, frame->height, kNoAllocMaxPixels);
  // the kernels run on the current device and read the volume's memory: the
  // two must be the same GPU (the scratch address is per device too)
  int device = 0;
  rf_status s = check_cuda(vol, cudaGetDevice(&device), "current device");
  if (s) return s;
  if (device != vol->device)
    return set_error(vol, RF_ERR_INVALID_ARG,
                     "rf_compute_mask_noalloc: current device %d is not the volume's device %d", device, vol->device);
  cudaError_t e;
  unsigned char* base = static_cast<unsigned char*>(mask_scratch_address(vol->device, &e));
  if (!base) return check_cuda(vol, e, "cudaGetSymbolAddress(mask scratch)");
  unsigned* ff = reinterpret_cast<unsigned*>(base + kNoAllocWordsOff);
  cudaStream_t st = (cudaStream_t)stream;
  const DevFrame f = make_dev_frame(frame);
  // the array keeps the previous call's contents: zero the words that count
  if ((s = check_cuda(vol, cudaMemsetAsync(ff, 0, sizeof(unsigned) * kFillWords, st), "scratch clear"))) return s;
  unsigned* tiles = reinterpret_cast<unsigned*>(base);
  if ((s = launch_seeds(vol, f, T_dev, tiles, ff, st))) return s;
  FillDesc d = make_fill_desc(vol, f, mask_dev);
  d.tiles = tiles;
  d.ff = ff;
  d.max_sweeps = d.max_sweeps < kNoAllocMaxSweeps ? d.max_sweeps : kNoAllocMaxSweeps;
  return launch_fill(vol, d, st);
}
