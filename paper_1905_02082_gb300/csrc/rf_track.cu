// Registration (ReFusion Sec. III-B) on sm_103a: Levenberg-Marquardt on the
// joint error of Eq. 4, E = sum_i V_SDF(exp(xi) T x_i)^2
//                         + w_c sum_i (V_I(exp(xi) T x_i) - I(p_i))^2,
// over three pixel sub-samplings (strides), coarse to fine.
//
// A whole registration (three levels, every LM iteration) is ONE cooperative
// launch of k_register, one CTA of 512 threads per SM.  At its start every
// thread writes the records of the pixels it will sample (camera point and
// intensity) into a per-volume buffer that only it reads again.  Per cost
// evaluation:
//   1. every thread takes its pixels' records: rigid transform, hash lookup of
//      the 8 lattice corners, trilinear SDF and intensity with analytic
//      gradients, residuals and Jacobians J = dV/dp [I | -[p]x] (left
//      perturbation), the SDF and the colour term side by side in packed FP32;
//   2. a warp-shuffle + shared-memory reduction of the 21 entries of J^T J,
//      the 6 of J^T r, the cost and the valid count gives one FP32 partial
//      per fixed chunk of pixels, written with the evaluation's tag;
//   3. EVERY CTA reads all partials, each until it carries the tag (this is
//      the only grid-wide wait, bounded), reduces them (FP32, the same fixed
//      order) and runs the same LM step on its shared-memory copy of the LM
//      state: accept or reject the candidate (mean cost E/N must decrease),
//      update lambda, solve the damped 6x6 system and compose the next
//      candidate pose exp(delta) T (FP32 with exactly formed residuals and a
//      pose carried as float pairs; see lm_candidate).  Identical inputs and
//      code give identical states in all CTAs, so no broadcast is needed: a
//      second hop through L2 costs more than the redundant step (one CTA
//      running the step and sending the pose to the others was measured at
//      123 us a 640x480 registration, this form at 102).
// A level ends early when the step falls below the thresholds.  Results are
// deterministic: fixed chunks, fixed pixel-to-thread mapping, fixed reduction
// order.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "rf_exchange.hpp"
#include "rf_queue.hpp"
#include "rf_volume.hpp"

namespace rf {
namespace {

// ---------------------------------------------------------------------------
// Packed FP32: one instruction works on two floats, here the SDF term (low)
// and the colour term (high) of a sample.  The registration issues about half
// as many arithmetic instructions this way; it is bound by instruction issue
// and latency, not by the FP32 pipes.
// ---------------------------------------------------------------------------
typedef unsigned long long f2;
__device__ __forceinline__ f2 pk(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpk(f2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// Normal equations of one thread's samples: the 21 entries of J^T J, the 6 of
// J^T r and the cost, each as (SDF sum, colour sum), and the valid count.
struct Acc {
  f2 v[28];
  float n;
};

__device__ __forceinline__ void clear(Acc& acc) {
#pragma unroll
  for (int i = 0; i < 28; ++i) acc.v[i] = 0ull;
  acc.n = 0.0f;
}

// The per-sample constants of a registration (uniform over the CTA).
struct SampleConst {
  float inv_voxel;
  float sdf_scale;   // stored SDF -> metres
  float gs_sdf;      // gradient of the stored SDF per voxel -> per metre
  float col_scale;   // stored intensity -> sqrt(w_c) times intensity
  float gs_col;      // its gradient
};

constexpr float kRound = 12582912.0f;  // 1.5 * 2^23: adding it leaves an integer in the low mantissa bits
constexpr float kBias = 8388608.0f;    // 2^23

// One sample: the pixel's camera point (x, y, z) and offset `off` (minus
// sqrt(w_c) times its intensity), looked up in the model at the pose `pose`
// (rows of R | t) and added to the normal equations when its 8 corners exist
// and were observed (corner n = dx + 2 dy + 4 dz); the colour term is added
// when all 8 also carry colour.  cached: the pixel's (key << 22 | pool) from
// an earlier sample, ~0 if none; returns the entry to keep when the block had
// to be looked up, else ~0.
//
// A third of the cells straddle a block border, and in most warps some lane's
// does.  All lanes therefore fetch their corners with the same eight loads
// from (pool, index) pairs; only the neighbour table's two loads are
// conditional.
template <int ST>
__device__ __forceinline__ unsigned long long add_sample(const DevVol& v, const SampleConst& c, const float4* pose,
                                                         float x, float y, float z, float off,
                                                         unsigned long long cached, Acc& acc) {
  const float4 r0 = pose[0], r1 = pose[1], r2 = pose[2];
  const float px = fmaf(r0.z, z, fmaf(r0.y, y, fmaf(r0.x, x, r0.w)));
  const float py = fmaf(r1.z, z, fmaf(r1.y, y, fmaf(r1.x, x, r1.w)));
  const float pz = fmaf(r2.z, z, fmaf(r2.y, y, fmaf(r2.x, x, r2.w)));
  const float qx = px * c.inv_voxel, qy = py * c.inv_voxel, qz = pz * c.inv_voxel;
  // floor: adding 1.5 * 2^23 rounded down leaves the integer in the low
  // mantissa bits (exact for |q| < 2^22)
  const float tx = __fadd_rd(qx, kRound), ty = __fadd_rd(qy, kRound), tz = __fadd_rd(qz, kRound);
  const int kx = __float_as_int(tx) - 0x4B400000, ky = __float_as_int(ty) - 0x4B400000,
            kz = __float_as_int(tz) - 0x4B400000;
  const float fx = qx - (tx - kRound), fy = qy - (ty - kRound), fz = qz - (tz - kRound);
  const int bx = kx >> 3, by = ky >> 3, bz = kz >> 3;
  // block coordinates from -kMaxCoord to kMaxCoord + 1 (no stored block has
  // the latter); larger |q|, infinities and NaN give k beyond +-2^21 above
  static_assert(kMaxCoord == 8191, "one comparison covers the three ranges");
  if ((unsigned)((bx + kMaxCoord) | (by + kMaxCoord) | (bz + kMaxCoord)) >= 16384u) return kEmpty;
  // the cached entry's upper 42 bits are the block key (bx, by, bz: 14 bits each)
  const unsigned khi = ((unsigned)bx << 18) | (((unsigned)by & 0x3FFFu) << 4) | (((unsigned)bz >> 10) & 15u);
  const unsigned klo = (unsigned)bz << 22;
  const unsigned chi = (unsigned)(cached >> 32), clo = (unsigned)cached;
  unsigned long long fresh = kEmpty;
  int pool;
  if (chi == khi && (clo ^ klo) < (1u << 22) && cached != kEmpty) {
    pool = (int)(clo & 0x3FFFFFu);  // same block as last time: no hash probe
  } else {
    pool = hash_find(v, bx, by, bz);
    if (pool < 0) return kEmpty;
    fresh = ((unsigned long long)khi << 32) | klo | (unsigned)pool;
  }
  const int lx = kx & 7, ly = ky & 7, lz = kz & 7;
  int a0 = pool, a1 = pool, a2 = pool, a3 = pool;  // pools of the corners at dx = 0: (dy, dz) = 00, 10, 01, 11
  int b0 = pool, b1 = pool, b2 = pool, b3 = pool;  // and at dx = 1
  if (((lx + 1) | (ly + 1) | (lz + 1)) & 8) {
    const int4 n0 = __ldg(v.nbr + 2 * (size_t)pool), n1 = __ldg(v.nbr + 2 * (size_t)pool + 1);
    const bool ex = lx == 7, ey = ly == 7, ez = lz == 7;
    const int m0 = ex ? n0.y : n0.x, m1 = ex ? n0.w : n0.z, m2 = ex ? n1.y : n1.x, m3 = ex ? n1.w : n1.z;
    a1 = ey ? n0.z : n0.x;
    a2 = ez ? n1.x : n0.x;
    a3 = ez ? (ey ? n1.z : n1.x) : a1;
    b0 = m0;
    b1 = ey ? m1 : m0;
    b2 = ez ? m2 : m0;
    b3 = ez ? (ey ? m3 : m2) : b1;
    if (min(min(min(a1, a2), min(a3, b0)), min(b1, min(b2, b3))) < 0) return fresh;
  }
  // FP32 storage: the uint2 words; FP16 storage: the 4-byte tracking words
  using Word = typename std::conditional<ST == RF_STORAGE_FP32, uint2, unsigned>::type;
  constexpr unsigned kStride = ST == RF_STORAGE_FP32 ? kBV : 2 * kBV;  // words per block
  const Word* words = reinterpret_cast<const Word*>(v.vox);
  const unsigned x1 = (unsigned)(lx + 1) & 7u, y0 = (unsigned)ly * 8u, y1 = ((unsigned)(ly + 1) & 7u) * 8u;
  const unsigned z0 = (unsigned)lz * 64u, z1 = ((unsigned)(lz + 1) & 7u) * 64u;
  Word w[8];  // (a 32-bit word index reaches every block: 2^22 blocks of 1,024 words)
  w[0] = __ldg(words + ((unsigned)a0 * kStride + (lx + y0 + z0)));
  w[1] = __ldg(words + ((unsigned)b0 * kStride + (x1 + y0 + z0)));
  w[2] = __ldg(words + ((unsigned)a1 * kStride + (lx + y1 + z0)));
  w[3] = __ldg(words + ((unsigned)b1 * kStride + (x1 + y1 + z0)));
  w[4] = __ldg(words + ((unsigned)a2 * kStride + (lx + y0 + z1)));
  w[5] = __ldg(words + ((unsigned)b2 * kStride + (x1 + y0 + z1)));
  w[6] = __ldg(words + ((unsigned)a3 * kStride + (lx + y1 + z1)));
  w[7] = __ldg(words + ((unsigned)b3 * kStride + (x1 + y1 + z1)));
  // corner pairs (SDF, intensity), the intensity with 2^23 added (exact: it is
  // a small integer), which cancels in the differences along x
  f2 d[4], e[4];  // differences along x, and values at fx, of the four x edges
  bool colour;
  {
    float I[8], F[8];
    if constexpr (ST == RF_STORAGE_FP32) {
      unsigned m = w[0].y;
#pragma unroll
      for (int n = 0; n < 8; ++n) {
        m = min(m, w[n].y);
        F[n] = __uint_as_float(w[n].x);
        I[n] = __uint_as_float(__dp2a_hi(722u, w[n].y, __dp2a_lo(2126u | (7152u << 16), w[n].y, 0x4B000000u)));
      }
      colour = m >= (1u << 24);  // the smallest colour weight (top byte) is not 0
    } else {
      unsigned m = 0u;
#pragma unroll
      for (int n = 0; n < 8; ++n) {
        const unsigned i8 = (w[n] >> 16) & 255u;  // intensity x 254; 255 marks a corner without colour
        m = max(m, i8);
        F[n] = __half2float(__ushort_as_half((unsigned short)(w[n] & 0xFFFFu)));
        I[n] = __uint_as_float(0x4B000000u | i8);
      }
      colour = m != 255u;
    }
    const f2 fx2 = pk(fx, fx), unbias = pk(-0.0f, -kBias);
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      const f2 p = pk(F[2 * n], I[2 * n]);
      d[n] = sub2(pk(F[2 * n + 1], I[2 * n + 1]), p);
      e[n] = fma2(fx2, d[n], add2(p, unbias));
    }
  }
  const f2 fy2 = pk(fy, fy), fz2 = pk(fz, fz);
  const f2 gy0 = sub2(e[1], e[0]), gy1 = sub2(e[3], e[2]);
  const f2 c0 = fma2(fy2, gy0, e[0]), c1 = fma2(fy2, gy1, e[2]);
  f2 gz = sub2(c1, c0);
  const f2 val = fma2(fz2, gz, c0);
  float V, I;
  unpk(val, V, I);
  // a never-observed corner stores NaN; every corner enters V, so one test
  // covers all eight
  if (V != V) return fresh;
  f2 gy = fma2(fz2, sub2(gy1, gy0), gy0);
  const f2 d0 = fma2(fy2, sub2(d[1], d[0]), d[0]), d1 = fma2(fy2, sub2(d[3], d[2]), d[2]);
  f2 gx = fma2(fz2, sub2(d1, d0), d0);
  const f2 gs = pk(c.gs_sdf, colour ? c.gs_col : 0.0f);
  gx = mul2(gx, gs);
  gy = mul2(gy, gs);
  gz = mul2(gz, gs);
  const f2 r = pk(ST == RF_STORAGE_FP32 ? V : V * c.sdf_scale, colour ? fmaf(I, c.col_scale, off) : 0.0f);
  f2 J[6];
  J[0] = gx;
  J[1] = gy;
  J[2] = gz;
  {
    // p x g, one half at a time: packing p twice costs more than it saves
    float ax, ay, az, bx, by, bz;
    unpk(gx, ax, bx);
    unpk(gy, ay, by);
    unpk(gz, az, bz);
    J[3] = pk(fmaf(py, az, -pz * ay), fmaf(py, bz, -pz * by));
    J[4] = pk(fmaf(pz, ax, -px * az), fmaf(pz, bx, -px * bz));
    J[5] = pk(fmaf(px, ay, -py * ax), fmaf(px, by, -py * bx));
  }
  int n = 0;
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = i; j < 6; ++j) {
      acc.v[n] = fma2(J[i], J[j], acc.v[n]);
      ++n;
    }
#pragma unroll
  for (int i = 0; i < 6; ++i) acc.v[21 + i] = fma2(J[i], r, acc.v[21 + i]);
  acc.v[27] = fma2(r, r, acc.v[27]);
  acc.n += 1.0f;
  return fresh;
}

// Geometry of one level: sampled pixels Ws x Hs, `chunk` of them per partial
// sum, and where its records start in the record buffer.
struct Level {
  int Ws, stride, npix, chunk, nchunks, rec0;
  unsigned long long magic;  // ceil(2^32 / Ws)
};

// State of a registration, one copy in the shared memory of every CTA.  Poses
// are rows (R | t) of four, as pairs of floats per entry (hi + lo, about 48
// bits; hi is the float pose an evaluation uses).
struct RegShared {
  Level level[3];
  int arrived;
  float sums[2][32];  // FP32 sums of an evaluation: 21 of J^T J, 6 of J^T r, cost, valid count; one slot holds the
                      // accepted pose's, the other the evaluation just reduced
  float4 pose[4][3];  // hi parts: the accepted pose, the candidate, and the two possible next candidates
  float plo[4][12];   // lo parts
  int stop[2][2];     // by parity of the evaluation: 1 when there is no next candidate (level converged) after an
                      // acceptance / a rejection
  int accept;
  float E;            // cost and valid count of the accepted pose
  unsigned N;
  double T0[12];      // the initial pose, returned unchanged when no candidate is accepted
  rf_track_info info;
};

// Packed index of entry (i, j), i <= j, of the upper triangle of a symmetric
// 6x6 matrix (row-major: the order of the 21 sums of J^T J).
__host__ __device__ constexpr int up6(int i, int j) { return i * 6 - i * (i - 1) / 2 + (j - i); }


__device__ __forceinline__ float rsqrt_approx(float x) {  // normal x
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// FP32 Cholesky factorisation of the damped matrix in place: A holds the
// upper triangle (row-major) on entry and L^T (L's column j stored as row j of
// the upper triangle) on exit; inv[j] = 1 / L[j][j] from the hardware
// reciprocal square root (the factor only preconditions the refined solve).
// False unless every pivot is positive and finite.  Right-looking (a pivot's
// updates of the trailing rows are independent of one another, so the chain
// from pivot to pivot is one reciprocal square root and three operations);
// constant bounds with guards unroll fully and keep A in registers.
__device__ __forceinline__ bool chol6(float A[21], float inv[6]) {
  bool ok = true;
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    const float s = A[up6(j, j)];
    ok = ok && (s > 0.0f) && (s < 3.0e38f);
    const float r = rsqrt_approx(fmaxf(s, 1.0e-30f));
    A[up6(j, j)] = s * r;
    inv[j] = r;
#pragma unroll
    for (int i = 0; i < 6; ++i)
      if (i > j) A[up6(j, i)] *= r;
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
      for (int k = 0; k < 6; ++k)
        if (i > j && k >= i) A[up6(i, k)] = fmaf(-A[up6(j, i)], A[up6(j, k)], A[up6(i, k)]);
  }
  return ok;
}

// Solves L L^T x = b in place (b -> x) with the factor of chol6 (FP32).
__device__ __forceinline__ void chol6_solve(const float A[21], const float inv[6], float b[6]) {
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    float t = b[i];
#pragma unroll
    for (int k = 0; k < 6; ++k)
      if (k < i) t = fmaf(-A[up6(k, i)], b[k], t);
    b[i] = t * inv[i];
  }
#pragma unroll
  for (int ii = 0; ii < 6; ++ii) {
    const int i = 5 - ii;
    float t = b[i];
#pragma unroll
    for (int k = 0; k < 6; ++k)
      if (k > i) t = fmaf(-A[up6(i, k)], b[k], t);
    b[i] = t * inv[i];
  }
}

// Error-free transformations (Knuth's TwoSum, the FMA form of Dekker's
// TwoProduct): a + b = s + e and a b = p + e exactly in FP32 arithmetic.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e) {
  p = a * b;
  e = fmaf(a, b, -p);
}

// a * na < b * nb, exactly, for finite floats a, b >= 0 and integers
// 0 <= na, nb < 2^32 (each product is a 56-bit integer times a power of two).
__device__ __forceinline__ bool prod_less(float a, unsigned na, float b, unsigned nb) {
  const unsigned ba = __float_as_uint(a), bb = __float_as_uint(b);
  const unsigned ea = (ba >> 23) & 255u, eb = (bb >> 23) & 255u;
  const unsigned long long P = (unsigned long long)((ba & 0x7FFFFFu) | (ea ? 0x800000u : 0u)) * na;
  const unsigned long long Q = (unsigned long long)((bb & 0x7FFFFFu) | (eb ? 0x800000u : 0u)) * nb;
  if (P == 0ull || Q == 0ull) return P == 0ull && Q != 0ull;
  const int xa = (int)(ea ? ea : 1u), xb = (int)(eb ? eb : 1u);  // exponent of the integer mantissa, + 150
  const int ta = 63 - __clzll((long long)P) + xa, tb = 63 - __clzll((long long)Q) + xb;
  if (ta != tb) return ta < tb;
  return xa >= xb ? (P << (xa - xb)) < Q : P < (Q << (xb - xa));
}

// The next candidate pose of the LM iteration, executed by the 32 lanes of one
// warp: solves (H + lambda diag H) d = -g for the sums of an evaluation at the
// pose (hi, lo) and writes exp(d) T to (out, out_lo).  Returns true when there
// is no next candidate: the step is below the thresholds or the solve failed.
//
// On GB300 a dependent FP64 instruction costs hundreds of cycles (measured
// with clock64 stamps in this loop: about 300-400 per dependent FP64
// operation), and the step lies on the registration's serial critical path;
// so the step works in FP32 and reaches FP64-class accuracy where it matters
// without FP64 latency:
//   solve: FP32 Cholesky, then one step of iterative refinement whose residual
//   -g - A d is formed exactly (FP32 error-free transformations: the products
//   of FP32 numbers and their sum carried to about 2^-46), which gives the
//   solution to the accuracy of an FP64 solve for the systems met here
//   (condition numbers ~10^2);
//   exp(d) - I = [A K + B K^2 | rho + B K rho + C K^2 rho] in FP32 (its
//   entries are of the order of the step, so FP32 is relative to the step);
//   the candidate pose T + (exp(d) - I) T: the increment in FP32, added
//   to the pose carried as float pairs with an error-free sum (lanes 0-11 in
//   parallel); the pair's high float is what the next evaluation uses.
// Not inlined: two warps call it (see register_body), and the instruction
// cache holds one copy.
__device__ __noinline__ bool lm_candidate(const float* sums, const float* hi, const float* lo, float lam, float eps_t2,
                                          float eps_r2, float* out, float* out_lo, int lane) {
  float A[21], inv[6], d[6], r[6];
#pragma unroll
  for (int q = 0; q < 21; ++q) A[q] = sums[q];
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    A[up6(i, i)] = fmaf(A[up6(i, i)], lam, A[up6(i, i)]);
    d[i] = -sums[21 + i];
  }
  const bool ok = chol6(A, inv);
  chol6_solve(A, inv, d);
  // residual -g - (H + lambda diag H) d, exact to about 2^-46: row i on
  // lane i, then gathered on every lane.  No branches (a divergent one per
  // column made this 1,000 of the step's 2,500 cycles): the damping term
  // lambda h_ii d_i is a seventh product.
  {
    const int i = lane < 6 ? lane : 0;
    const int row = up6(i, i) - i;  // entry (i, j), j >= i, at row + j
    float sh = -sums[21 + i], sl = 0.0f, hii = 0.0f, di = 0.0f;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      const float h = sums[i <= j ? row + j : up6(j, j) - j + i];
      hii = i == j ? h : hii;
      di = i == j ? d[j] : di;
      float p, pe, e;
      two_prod(h, d[j], p, pe);
      two_sum(sh, -p, sh, e);
      sl += e - pe;
    }
    float lh, lhe, p, pe, e;
    two_prod(lam, hii, lh, lhe);
    two_prod(lh, di, p, pe);
    two_sum(sh, -p, sh, e);
    sl += e - pe - lhe * di;
    const float ri = sh + sl;
#pragma unroll
    for (int q = 0; q < 6; ++q) r[q] = __shfl_sync(0xffffffffu, ri, q);
  }
  chol6_solve(A, inv, r);
#pragma unroll
  for (int q = 0; q < 6; ++q) d[q] += r[q];  // the refined step
  const float nr2 = fmaf(d[0], d[0], fmaf(d[1], d[1], d[2] * d[2]));
  const float p0 = d[3], p1 = d[4], p2 = d[5];
  const float t2 = fmaf(p0, p0, fmaf(p1, p1, p2 * p2));
  if (!ok || !(nr2 < 3.0e38f) || !(t2 < 3.0e38f) || (nr2 < eps_t2 && t2 < eps_r2)) return true;
  // exponential map minus identity: A, B, C of theta^2
  float cA, cB, cC;
  if (t2 < 0.01f) {  // Taylor series in theta^2, enough terms for FP32 below theta = 0.1
    cA = fmaf(t2, fmaf(t2, fmaf(t2, -1.0f / 5040.0f, 1.0f / 120.0f), -1.0f / 6.0f), 1.0f);
    cB = fmaf(t2, fmaf(t2, fmaf(t2, -1.0f / 40320.0f, 1.0f / 720.0f), -1.0f / 24.0f), 0.5f);
    cC = fmaf(t2, fmaf(t2, fmaf(t2, -1.0f / 362880.0f, 1.0f / 5040.0f), -1.0f / 120.0f), 1.0f / 6.0f);
  } else {
    const float th = sqrtf(t2);
    float sn, cs;
    sincospif(th * 0.318309886183790672f, &sn, &cs);  // argument reduction by pi is exact
    cA = sn / th;
    cB = (1.0f - cs) / t2;
    cC = (th - sn) / (t2 * th);
  }
  // increment (exp(d) - I) T in FP32 from the float pose, added to the pose
  // carried as float pairs (lanes 0-11: rows 0-2, columns 0-3).  Row i of
  // exp(d) - I: Er = A K + B K^2 with K v = phi x v and K^2 = phi phi^T -
  // theta^2 I; et = rho + B K rho + C K^2 rho.
  const int at = lane < 12 ? lane : 0;
  const int i = at >> 2, j = at & 3;
  const float h0 = hi[j], h1 = hi[4 + j], h2 = hi[8 + j], hT = hi[at], lT = lo[at];
  const float pi = i == 0 ? p0 : (i == 1 ? p1 : p2);
  // row i of K: (K_i0, K_i1, K_i2)
  const float k0 = i == 0 ? 0.0f : (i == 1 ? p2 : -p1);
  const float k1 = i == 0 ? -p2 : (i == 1 ? 0.0f : p0);
  const float k2 = i == 0 ? p1 : (i == 1 ? -p0 : 0.0f);
  const float e0 = fmaf(cA, k0, cB * fmaf(pi, p0, i == 0 ? -t2 : 0.0f));
  const float e1 = fmaf(cA, k1, cB * fmaf(pi, p1, i == 1 ? -t2 : 0.0f));
  const float e2 = fmaf(cA, k2, cB * fmaf(pi, p2, i == 2 ? -t2 : 0.0f));
  float inc = fmaf(e0, h0, fmaf(e1, h1, e2 * h2));
  // column 3: + (rho + B K rho + C K^2 rho)_i
  const float kr = fmaf(k0, d[0], fmaf(k1, d[1], k2 * d[2]));  // (K rho)_i
  const float kr0 = p1 * d[2] - p2 * d[1], kr1 = p2 * d[0] - p0 * d[2], kr2 = p0 * d[1] - p1 * d[0];
  const float kk = fmaf(k0, kr0, fmaf(k1, kr1, k2 * kr2));  // (K K rho)_i
  const float rho_i = i == 0 ? d[0] : (i == 1 ? d[1] : d[2]);
  const float trans = fmaf(cC, kk, fmaf(cB, kr, rho_i));
  inc += j == 3 ? trans : 0.0f;
  float sum, err;
  two_sum(hT, inc, sum, err);
  err += lT;
  const float hn = sum + err;  // renormalised: hn is the nearest float of the pair's sum
  if (lane < 12) {
    out[lane] = hn;
    out_lo[lane] = err - (hn - sum);
  }
  return false;
}

constexpr int kRegThreads = 512;
constexpr int kRegWarps = kRegThreads / 32;
// Steps (a chunk per slot each) between CTA barriers in a batch, where a CTA
// has several chunks: the warps of a CTA need not keep step with its slowest
// one at each.  A warp per chunk then sums the warps' partials (at most 4 slots
// x 4 steps).
constexpr int kBatchSteps = 4;

// Pixels per partial sum: a fixed chunk of the sampled pixels of a level, a
// function of their number only, so the partials, and thus the result, do not
// depend on how many CTAs run the registration.  At most kRegChunks chunks
// (one per CTA of a registration that has the GPU to itself, 98.7 % of the
// SMs), of at least 128 pixels and a whole number of warps.
__host__ __device__ __forceinline__ int chunk_pixels(int npix) {
  const int c = ((npix + kRegChunks - 1) / kRegChunks + 127) & ~127;
  return c > 128 ? c : 128;
}

// Position in the frame of sample i of a level (row = i / Ws by a reciprocal
// multiply, off by at most one for i < 2^32, then corrected).
__device__ __forceinline__ void locate(const Level& L, int i, int& u, int& v) {
  int row = (int)(((unsigned long long)i * L.magic) >> 32);
  if (row * L.Ws > i) --row;
  else if ((row + 1) * L.Ws <= i) ++row;
  u = (i - row * L.Ws) * L.stride;
  v = row * L.stride;
}
__device__ __forceinline__ int pixel_of_sample(const Level& L, int W, int i) {
  if (L.stride == 1) return i;
  int u, v;
  locate(L, i, u, v);
  return v * W + u;
}

// Record of sample i of a level, written once per registration by the thread
// that samples it: camera point of Eq. 1 and minus sqrt(w_c) times the
// intensity; z = 0 where the pixel is not sampled (invalid depth or masked).
__device__ __forceinline__ void write_record(const RegDesc& d, const Level& L, float col_off, int i) {
  const DevFrame& f = d.f;
  int u, v;
  locate(L, i, u, v);
  const int idx = v * f.W + u;
  unsigned raw = __ldg(f.depth + idx);
  if (d.mask && __ldg(d.mask + idx)) raw = 0u;
  const uint8_t* cp = f.rgb + 3 * (size_t)idx;
  const unsigned rgb = (unsigned)__ldg(cp) | ((unsigned)__ldg(cp + 1) << 8) | ((unsigned)__ldg(cp + 2) << 16);
  float4 r = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  if (pixel_valid(d.p, raw)) {
    const float D = u2f_exact(raw) * d.p.inv_depth_scale;
    r.x = (u2f_exact((unsigned)u) - f.cx) * f.ifx * D;
    r.y = (u2f_exact((unsigned)v) - f.cy) * f.ify * D;
    r.z = D;
    r.w = rgb_intensity_raw(rgb) * col_off;
  }
  d.rec[L.rec0 + i] = r;
}

// The counts' memory operations (rf_exchange.hpp) on the device.
struct CountMem {
  __device__ void red_relaxed(unsigned* p, unsigned v) { red_relaxed_gpu_add(p, v); }
  __device__ unsigned add_acq_rel(unsigned* p, unsigned v) {
    unsigned old;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
  }
};

// Every CTA of a registration group calls this once, after its last use of
// the exchange.  The last CTA to leave clears the arrival count and advances
// the tag base past the
// registration's tags (at most 3 + the sum of the level iteration caps); when
// the tags would reach kTagLimit it first clears the whole partial buffer,
// whose tags then all read 0, and restarts the base at 0.  Either way every
// tag left in the buffer is below the next registration's tags.
__device__ __forceinline__ void leave_registration(const RegDesc& d, int G, unsigned tag0) {
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    CountMem mem;
    s_last = last_to_leave(mem, d.tags + 1, (unsigned)G);
  }
  __syncthreads();
  if (!s_last) return;
  const unsigned span = (unsigned)(d.c.iters[0] + d.c.iters[1] + d.c.iters[2] + 3);
  unsigned next = tag0 + span;
  if (next >= kTagLimit - span) {
    const int n = 2 * kRegWords * d.max_slots;
    for (int i = threadIdx.x; i < n; i += kRegThreads) d.partials[i] = make_ulonglong2(0ull, 0ull);
    next = 0u;
  }
  if (threadIdx.x == 0) {
    d.tags[2] = 0u;
    d.tags[1] = 0u;
    d.tags[0] = next;
  }
}

// One whole registration (see the file comment) run by a group of G CTAs,
// this CTA being number lb of the group.
//
// Exchange of the partial sums: evaluation e of the registration tags its
// partials with base + e + 1 (base: d.tags[0]) and then counts the CTA in
// d.tags[2] with a relaxed reduction; every CTA waits until the count shows
// (nearly) all G arrivals of e, then reads the partials, re-polling any word
// that does not carry the tag yet (no fence orders a CTA's partials before its
// count, so the tags carry the ordering).  Where every CTA of a large group
// has a chunk the last eighth of the arrivals is not waited for: the reads' round trip then
// passes while the slowest CTAs finish (640x480 registration 108.7 -> 104.2
// us, 1280x720 213.6 -> 206.1; with no count at all the polling readers slow
// those CTAs down: 220.2).  Double buffering by evaluation parity is safe: a
// CTA writes evaluation e + 2 only after it has read the words of e + 1 of
// every CTA that has a chunk, and, where some CTA has none, after all G CTAs
// arrived at e + 1; a CTA does either only after it has read all of e.
//
// Little of the LM step follows the reduction: while the CTA waits for the
// others, one of its warps computes the next candidate of a rejection (it
// needs the accepted pose's sums only); after the reduction warp 0 computes
// the next candidate of an acceptance while another warp decides which of the
// two applies.  The first of them shares warp 0's scheduler and so leaves its
// instruction cache holding the step's code.
template <int ST, int kStepsPerBarrier>
__device__ __forceinline__ void register_body(const RegDesc& d, int lb, int G) {
  __shared__ RegShared S;
  __shared__ float red[2][kStepsPerBarrier][kRegWarps][32];  // per-warp sums of chunks, double-buffered
  constexpr int kRejectWarp = 12, kDecideWarp = 13;
  CountMem count;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const DevFrame& f = d.f;

  if (threadIdx.x < 3) {
    const int l = threadIdx.x;
    int rec0 = 0;
    Level L;
    for (int i = 0; i <= l; ++i) {
      L.rec0 = rec0;
      L.stride = d.c.strides[i];
      L.Ws = (f.W + L.stride - 1) / L.stride;
      L.npix = L.Ws * ((f.H + L.stride - 1) / L.stride);
      rec0 += L.npix;
    }
    L.chunk = chunk_pixels(L.npix);
    L.nchunks = (L.npix + L.chunk - 1) / L.chunk;
    L.magic = (0x100000000ull + L.Ws - 1) / L.Ws;
    S.level[l] = L;
  }
  if (threadIdx.x == 32) {
    rf_track_info z = {};
    S.info = z;
    S.E = 0.0f;
    S.N = 0u;
  }
  if (threadIdx.x >= 64 && threadIdx.x < 76) {  // the initial pose as float pairs (FP64 once per registration)
    const int q = threadIdx.x - 64;
    const double t = d.T_init[q];
    S.T0[q] = t;
    const float hi = (float)t;
    reinterpret_cast<float*>(S.pose[0])[q] = hi;
    S.plo[0][q] = (float)(t - (double)hi);
  }
  SampleConst c;
  {
    const float swc = sqrtf(d.p.w_c);
    c.inv_voxel = d.p.inv_voxel;
    c.sdf_scale = ST == RF_STORAGE_FP32 ? 1.0f : d.p.tau;  // FP16 storage holds F / tau
    c.gs_sdf = d.p.inv_voxel * c.sdf_scale;
    c.col_scale = (ST == RF_STORAGE_FP32 ? kIntensityScale : kI8Scale) * swc;
    c.gs_col = c.col_scale * d.p.inv_voxel;
  }
  __syncthreads();
  const unsigned tag0 = ld_relaxed_gpu(d.tags);  // written by the previous registration's last CTA

  // chunks narrower than the CTA run side by side, one per warp group (slot):
  // chunk lb + G (slot + slots step) at each step
  int chunk = 0, nchunks = 0, npix = 0, width = 1, slots = 1, slot = 0, tin = 0;
  auto set_level = [&](const Level& L) {
    chunk = L.chunk;
    nchunks = L.nchunks;
    npix = L.npix;
    width = min(chunk, kRegThreads);  // threads per chunk
    slots = kRegThreads / width;
    slot = threadIdx.x / width;
    tin = threadIdx.x - slot * width;
  };
  // this thread's samples of a chunk: first, first + width, ... below end
  auto bounds = [&](int ch, int& end) {
    end = slot < slots && ch < nchunks ? min(npix, (ch + 1) * chunk) : 0;
    return ch * chunk + tin;
  };
  {
    const float col_off = -kIntensityScale * sqrtf(d.p.w_c);
    for (int l = 0; l < 3; ++l) {
      set_level(S.level[l]);
      for (int ch = lb + G * slot; ch < nchunks && slot < slots; ch += G * slots) {
        int end;
        for (int i = bounds(ch, end); i < end; i += width) write_record(d, S.level[l], col_off, i);
      }
    }
  }

  unsigned eval = 0;
  bool failed = false, moved = false;
  int iT = 0, iC = 1, iA = 2, iR = 3;  // pose slots: accepted, candidate, next after acceptance, next after rejection
  int cur = 0;                         // slot of S.sums that holds the accepted pose's
  Acc acc;                             // empty between the steps
  clear(acc);
  for (int l = 0; l < 3 && !failed; ++l) {
    const Level& L = S.level[l];
    const float4* records = d.rec + L.rec0;
    set_level(L);
    const int iters = d.c.iters[l];
    // the next sample's record and cached block entry
    float4 rec = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    unsigned long long cached = kEmpty;
    auto fetch = [&](int i) {
      rec = records[i];
      cached = d.pxcache[pixel_of_sample(L, f.W, i)];
    };
    {
      int end;
      const int i = bounds(lb + G * slot, end);
      if (i < end) fetch(i);
    }
    const unsigned slack = G >= 64 && nchunks >= G && d.bar_extra == 0u ? (unsigned)G / 8u : 0u;
    bool done = false;
    int k = 0;  // damping lambda0 10^k: rejections minus acceptances
    for (int it = 0; it <= iters && !done; ++it) {
      const bool first = it == 0, last = it == iters;
      const float4* pose = S.pose[first ? iT : iC];
      ulonglong2* part = d.partials + (size_t)(eval & 1u) * kRegWords * d.max_slots;
      const unsigned tag = tag0 + eval + 1u;
      int par = 0;
      for (int step0 = 0; lb + G * slots * step0 < nchunks; step0 += kStepsPerBarrier) {
        for (int sb = 0; sb < kStepsPerBarrier && lb + G * slots * (step0 + sb) < nchunks; ++sb) {
          const int ch = lb + G * (slot + slots * (step0 + sb));
          int end;
          int i = bounds(ch, end);
          const bool any = __any_sync(0xffffffffu, i < end);
#pragma unroll 1
          while (i < end) {
            const float4 r = rec;
            const unsigned long long cj = cached;
            const int here = i;
            i += width;
            if (i < end) fetch(i);  // the next sample's record
            if (r.z > 0.0f) {
              const unsigned long long fresh = add_sample<ST>(d.v, c, pose, r.x, r.y, r.z, r.w, cj, acc);
              if (fresh != kEmpty) d.pxcache[pixel_of_sample(L, f.W, here)] = fresh;
            }
          }
          // chunk partial: a butterfly over the warp that halves the vector at
          // every step (31 shuffles for 32 slots) and leaves component c on
          // lane c, then the warps in fixed order
          float* mine = &red[par][sb][warp][lane];
          if (any) {
            __syncwarp();
            float v[32];
#pragma unroll
            for (int q = 0; q < 28; ++q) {
              float a, b;
              unpk(acc.v[q], a, b);
              v[q] = a + b;
            }
            v[28] = acc.n;
            v[29] = v[30] = v[31] = 0.0f;
#pragma unroll
            for (int h = 16; h > 0; h >>= 1) {
              const bool upper = (lane & h) != 0;
#pragma unroll
              for (int q = 0; q < h; ++q) {
                const float keep = upper ? v[q + h] : v[q];
                const float send = upper ? v[q] : v[q + h];
                v[q] = keep + __shfl_xor_sync(0xffffffffu, send, h);
              }
            }
            *mine = v[0];
          } else {
            *mine = 0.0f;
          }
          clear(acc);
          if (lb + G * slots * (step0 + sb + 1) < nchunks) {  // (the last step's follows below, after its partial)
            const int j = bounds(ch + G * slots, end);
            if (j < end) fetch(j);
          }
        }
        __syncthreads();
        // the chunk partials: the warps' sums of each in order; lane w < 10
        // writes components 3 w .. 3 w + 2 with the tag.  No barrier after
        // it: the next steps write the other buffer, and this one again only
        // after their barrier, which these reads precede.
        const int sb = warp / slots, cs = lb + G * (warp - sb * slots + slots * (step0 + sb));
        if (sb < kStepsPerBarrier && cs < nchunks) {
          const int wpc = width / 32;
          const float* from = &red[par][sb][(warp - sb * slots) * wpc][lane];
          float t[kRegWarps], sv = 0.0f;
#pragma unroll
          for (int w = 0; w < kRegWarps; ++w) t[w] = w < wpc ? from[32 * w] : 0.0f;
#pragma unroll
          for (int w = 0; w < kRegWarps; ++w) sv += t[w];
          const unsigned s0 = __float_as_uint(__shfl_sync(0xffffffffu, sv, (3 * lane) & 31));
          const unsigned s1 = __float_as_uint(__shfl_sync(0xffffffffu, sv, (3 * lane + 1) & 31));
          const unsigned s2 = __float_as_uint(__shfl_sync(0xffffffffu, sv, (3 * lane + 2) & 31));
          if (lane < kRegWords) st_relaxed_gpu_b128(part + lane * d.max_slots + cs, s0, s1, s2, tag);
        }
        par ^= 1;
      }
      if (lb < nchunks) {
        // arrival: one relaxed count per CTA (other warps' partial stores may
        // still be on their way: the readers check the tags)
        if (threadIdx.x == 0) arrive(count, d.tags + 2);
        // for the next evaluation, which samples the same pixels, during the
        // exchange: the first record
        int end;
        const int j = bounds(lb + G * slot, end);
        if (j < end) fetch(j);
      }
      if (lb >= nchunks && threadIdx.x == 0) arrive(count, d.tags + 2);
      if (threadIdx.x == 0)
        S.arrived = await_count(d.tags + 2, (eval + 1u) * (unsigned)G + d.bar_extra - slack, d.spin_limit);
      // meanwhile: the next candidate should this one be rejected
      if (warp == kRejectWarp && !first && !last) {
        const bool stop = lm_candidate(S.sums[cur], reinterpret_cast<const float*>(S.pose[iT]), S.plo[iT],
                                       d.c.lambda_pow[min(k + 1, kLambdaPow) + kLambdaPow], d.c.eps_t2f, d.c.eps_r2f,
                                       reinterpret_cast<float*>(S.pose[iR]), S.plo[iR], lane);
        if (lane == 0) S.stop[eval & 1u][1] = stop;
      }
      __syncthreads();
      // FP32 reduction of the chunk partials in a fixed order (lane-strided
      // sums, then a shuffle tree), one warp per word of three components;
      // words without this evaluation's tag are read again, all together,
      // until they have it
      bool ok = S.arrived != 0;
      float* sums = S.sums[cur ^ 1];
      if (warp < kRegWords && ok) {
        const ulonglong2* row = part + warp * d.max_slots;
        constexpr int kLoads = (kRegChunks + 31) / 32;
        ulonglong2 w[kLoads];
#pragma unroll
        for (int u = 0; u < kLoads; ++u) w[u] = make_ulonglong2(0ull, (unsigned long long)~tag << 32);
        long long spins = 0;
        for (;;) {
          bool here = true;
#pragma unroll
          for (int u = 0; u < kLoads; ++u)
            if (lane + 32 * u < nchunks && (unsigned)(w[u].y >> 32) != tag)
              w[u] = ld_relaxed_gpu_b128(row + lane + 32 * u);
#pragma unroll
          for (int u = 0; u < kLoads; ++u)
            here = here && (lane + 32 * u >= nchunks || (unsigned)(w[u].y >> 32) == tag);
          if (__all_sync(0xffffffffu, here)) break;
          if (++spins > d.spin_limit) {
            ok = false;
            break;
          }
          if (spins > 4096) __nanosleep(64);
        }
        float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f;
#pragma unroll
        for (int u = 0; u < kLoads; ++u) {
          if (lane + 32 * u < nchunks) {
            s0 += __uint_as_float((unsigned)w[u].x);
            s1 += __uint_as_float((unsigned)(w[u].x >> 32));
            s2 += __uint_as_float((unsigned)w[u].y);
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          s0 += __shfl_down_sync(0xffffffffu, s0, o);
          s1 += __shfl_down_sync(0xffffffffu, s1, o);
          s2 += __shfl_down_sync(0xffffffffu, s2, o);
        }
        if (lane == 0) {
          sums[3 * warp] = s0;
          sums[3 * warp + 1] = s1;
          sums[3 * warp + 2] = s2;
        }
      }
      if (!__syncthreads_and(ok)) {  // some wait ran out: leave, reporting it once per CTA
        if (threadIdx.x == 0) atomicOr(d.status, ST_BARRIER);
        failed = true;
        break;
      }
      // The LM step.  First evaluation of a level (at the accepted pose):
      // always taken.  Later ones: the candidate is accepted when the mean
      // cost decreases (En/Nn < E/N, compared exactly as En N < E Nn on the
      // integer mantissas).
      if (warp == 0 && !last) {
        const int from = first ? iT : iC;
        const int ka = first ? 0 : max(k - 1, -kLambdaPow);
        const bool stop = lm_candidate(sums, reinterpret_cast<const float*>(S.pose[from]), S.plo[from],
                                       d.c.lambda_pow[ka + kLambdaPow], d.c.eps_t2f, d.c.eps_r2f,
                                       reinterpret_cast<float*>(S.pose[iA]), S.plo[iA], lane);
        if (lane == 0) S.stop[eval & 1u][0] = stop;
      }
      if (warp == kDecideWarp && lane == 0) {
        const float En = sums[27];
        const unsigned Nn = (unsigned)(sums[28] + 0.5f);  // exact up to 2^24 samples, then rounded as a float
        const bool enough = (long long)Nn >= d.c.min_valid;
        const bool accept = first || (enough && prod_less(En, S.N, S.E, Nn));
        S.info.evals++;
        S.info.level_evals[l]++;
        if (accept) {
          S.E = En;
          S.N = Nn;
        }
        S.accept = accept ? (first && !enough ? 2 : 1) : 0;  // 2: too few pixels, the level ends
      }
      __syncthreads();
      // every thread follows the decision: slots and damping
      const int accept = S.accept;
      const bool converged = accept != 2 && !last && S.stop[eval & 1u][accept ? 0 : 1] != 0;
      if (accept) {
        cur ^= 1;
        k = first ? 0 : max(k - 1, -kLambdaPow);
        moved = moved || !first;
        const int t = first ? iC : iT;  // the slot that is free now
        if (!first) iT = iC;
        iC = iA;
        iA = t;
      } else {
        k = min(k + 1, kLambdaPow);
        const int t = iC;
        iC = iR;
        iR = t;
      }
      ++eval;
      done = accept == 2 || converged;
      if (converged && threadIdx.x == 0) S.info.converged[l] = 1;
    }
  }
  leave_registration(d, G, tag0);
  if (failed || lb != 0) return;
  if (threadIdx.x < 16) {  // the pose in FP64: hi + lo of each entry, the last row 0 0 0 1
    const int q = threadIdx.x;
    double t = q == 15 ? 1.0 : 0.0;
    if (q < 12) t = moved ? (double)reinterpret_cast<const float*>(S.pose[iT])[q] + (double)S.plo[iT][q] : S.T0[q];
    d.T_out[q] = t;
  }
  if (threadIdx.x == 0 && d.info) {
    rf_track_info out = S.info;
    out.final_cost = S.N > 0u ? (double)S.E / (double)S.N : 0.0;
    out.final_valid = (int64_t)S.N;
    *d.info = out;
  }
}

// One registration on the whole grid.
template <int ST>
__global__ void __launch_bounds__(kRegThreads, 1) k_register(RegDesc d) {
  register_body<ST, 1>(d, blockIdx.x, gridDim.x);
}

// The queue's memory operations (rf_queue.hpp) on the device: relaxed, at GPU
// scope (the words carry all that they tell).
struct QueueMem {
  const RegDesc* descs;
  const int* order;
  __device__ unsigned load(const unsigned* p) { return ld_relaxed_gpu(p); }
  __device__ unsigned add(unsigned* p, unsigned v) { return atomicAdd(p, v); }
  __device__ unsigned cas(unsigned* p, unsigned expected, unsigned v) { return atomicCAS(p, expected, v); }
  __device__ void pause(long long spins) {
    if (spins > 4096) __nanosleep(64);
  }
  __device__ void abandon(int at) { atomicOr(descs[order[at]].status, ST_BARRIER); }
};

__device__ __noinline__ int next_stream(const RegDesc* descs, const RegQueue& q, int at, bool leader, long long limit) {
  QueueMem mem = {descs, q.order};
  return leader ? queue_lead(mem, q.links, q.counter, q.groups_left, at, *q.length)
                : queue_follow(mem, q.links, at, *q.length, limit);
}

// The registrations of a batch in one cooperative launch.  CTA b is member
// b - first[g] of group g = cta_group[b] (-1: no work) of first[g + 1] -
// first[g] CTAs; groups never wait on each other.  A group registers the
// streams of the queue one after the other (rf_queue.hpp).
// Streams need 12 to 23 evaluations and have up to 12 times the pixels of
// others; with a fixed set of streams per launch a quarter of the SMs' time was
// spent waiting for the launch's last stream.  The queue and its counters
// are part of the table that each call uploads.
template <int ST>
__global__ void __launch_bounds__(kRegThreads, 1) k_register_batch(const RegDesc* __restrict__ descs,
                                                                   const __grid_constant__ RegQueue q) {
  __shared__ RegDesc sd;
  __shared__ int s_at;
  const int g = q.cta_group[blockIdx.x];
  if (g < 0) return;
  const int lb = blockIdx.x - q.first[g], G = q.first[g + 1] - q.first[g];
  for (bool begun = false;; begun = true) {
    if (threadIdx.x == 0)  // (there are no more groups than streams)
      s_at = begun ? next_stream(descs, q, s_at, lb == 0, sd.spin_limit) : g;
    __syncthreads();
    if (s_at >= *q.length) return;
    const RegDesc* from = descs + q.order[s_at];
    static_assert(sizeof(RegDesc) % 4 == 0, "copied in words");
    for (unsigned i = threadIdx.x; i < sizeof(RegDesc) / 4; i += kRegThreads)
      reinterpret_cast<unsigned*>(&sd)[i] = reinterpret_cast<const unsigned*>(from)[i];
    __syncthreads();
    register_body<ST, kBatchSteps>(sd, lb, G);
    __syncthreads();
  }
}

}  // namespace

int register_max_grid(int device) {
  // the smallest residency over the kernels launched with this grid
  const void* fns[] = {(const void*)k_register<RF_STORAGE_FP32>, (const void*)k_register<RF_STORAGE_FP16>,
                       (const void*)k_register_batch<RF_STORAGE_FP32>, (const void*)k_register_batch<RF_STORAGE_FP16>};
  int per_sm = 1 << 20, sms = 0;
  for (const void* fn : fns) {
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, kRegThreads, 0);
    per_sm = n < per_sm ? n : per_sm;
  }
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  return per_sm * sms;
}

RegDesc make_reg_desc(rf_volume* vol, const DevFrame& f, const double* T_init, const uint8_t* mask, double* T_out,
                      rf_track_info* info) {
  RegDesc d;
  d.v = vol->dv;
  d.f = f;
  d.p = vol->dp;
  d.mask = mask;
  d.T_init = T_init;
  d.T_out = T_out;
  d.info = info;
  d.c.lambda0 = vol->p.lm_lambda0;
  d.c.eps_t = vol->p.lm_eps_trans;
  d.c.eps_r = vol->p.lm_eps_rot;
  d.c.eps_t2f = (float)(vol->p.lm_eps_trans * vol->p.lm_eps_trans);
  d.c.eps_r2f = (float)(vol->p.lm_eps_rot * vol->p.lm_eps_rot);
  for (int k = -kLambdaPow; k <= kLambdaPow; ++k)
    d.c.lambda_pow[k + kLambdaPow] = (float)(vol->p.lm_lambda0 * std::pow(10.0, (double)k));
  d.c.min_valid = vol->p.lm_min_valid;
  for (int l = 0; l < 3; ++l) {
    d.c.iters[l] = vol->p.lm_iters[l];
    d.c.strides[l] = vol->p.lm_strides[l];
  }
  d.partials = vol->d_partials;
  d.max_slots = vol->max_slots;
  d.tags = vol->d_regtags;
  d.status = vol->d_status;
  d.spin_limit = vol->wait_spins;
  d.bar_extra = vol->wait_extra;
  d.pxcache = vol->d_pxcache;
  d.rec = reinterpret_cast<float4*>(vol->d_cand);
  return d;
}

static rf_status launch_coop(rf_volume* vol, const void* fn, int grid, void** args, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kRegThreads);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return check_cuda(vol, cudaLaunchKernelExC(&cfg, fn, args), "registration launch");
}

rf_status launch_track(rf_volume* vol, const DevFrame& f, const double* T_init, const uint8_t* mask, double* T_out,
                       rf_track_info* info, cudaStream_t st) {
  RegDesc d = make_reg_desc(vol, f, T_init, mask, T_out, info);
  void* args[] = {&d};
  const void* fn = vol->p.storage == RF_STORAGE_FP16 ? (const void*)k_register<RF_STORAGE_FP16>
                                                     : (const void*)k_register<RF_STORAGE_FP32>;
  // no more CTAs than the finest level has chunks: then every CTA has pixels
  // at every level of more than kRegChunks * 128 samples (see register_body)
  int most = 1;
  for (int l = 0; l < 3; ++l) {
    const int s = vol->p.lm_strides[l], n = ((f.W + s - 1) / s) * ((f.H + s - 1) / s), c = chunk_pixels(n);
    most = std::max(most, (n + c - 1) / c);
  }
  return launch_coop(vol, fn, std::min(vol->reg_grid, most), args, st);
}

rf_status launch_register_batch(rf_volume* vol, const RegDesc* descs, const RegQueue& q, int total_ctas,
                                cudaStream_t st) {
  RegQueue a = q;
  void* args[] = {(void*)&descs, (void*)&a};
  const void* fn = vol->p.storage == RF_STORAGE_FP16 ? (const void*)k_register_batch<RF_STORAGE_FP16>
                                                     : (const void*)k_register_batch<RF_STORAGE_FP32>;
  return launch_coop(vol, fn, total_ctas, args, st);
}

}  // namespace rf
