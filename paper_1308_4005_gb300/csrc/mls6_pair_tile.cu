// Local part of the split (Eq. g_0), tile form (pair_split 2048, FP32 and
// mixed plans): a warp evaluates 8 consecutive cell-sorted atoms against the
// candidates near any of them.
//
// The per-atom kernel is bound by instruction issue with half its lanes idle:
// the lanes of a warp walk different candidate lists in lockstep, and the
// pair arithmetic runs whenever any lane has a hit.  Here the warp works
// through one list for its 8 atoms:
//   - no lane waits for another: every loop bound is uniform over the warp;
//   - a candidate is loaded, and tested against the atoms' bounding box, once
//     for all 8 (about 1 in 3 pairs of a candidate that passes lies inside
//     the cutoff);
//   - the pair arithmetic is packed FP32, two candidates per instruction
//     (add/mul/fma.rn.f32x2; each half rounds as the scalar instruction).
// A pair outside the cutoff is evaluated at r = a, where both sums below
// vanish, so it needs no mask; the atom itself (r = 0) is moved there too.
//
// Steps of a warp, for each segment of its atoms that shares a row of cells:
//   1. lane t sets up neighbour row t: skipped if its y-z distance from the
//      segment's bounding box is >= a, else clipped in x, and split into
//      runs of one periodic image; the runs go to a table, those of the zero
//      image apart from the others;
//   2. the runs are read as one stream, 32 candidates at a time; those within
//      a of the bounding box are compacted into a list in shared memory;
//   3. the list is evaluated 32 candidates at a time: lane = 2 atoms x 4
//      candidates (4 lane groups of atoms x 8 of candidates), the candidates
//      read as two packed pairs per coordinate;
//   4. the sums are added over the candidate groups by a transposing tree.
// The list and the trees have a fixed order: results are reproducible bit for
// bit.
//
// What bounds it (1,048,576 atoms, density 0.85, a = 3): 494 candidates and 298
// listed ones per warp; about 60% of the issue slots and of the FP32 pipe busy
// (a packed instruction holds the pipe for two cycles).  Of the time about a
// fifth sets up rows, a quarter lists, the rest evaluates, at 58 cycles per
// packed pair against 48 of its 24 packed instructions alone.  8 atoms per warp
// and 2 x 4 per lane: 4 atoms leave less arithmetic (2.3 against 3.4 slots per
// pair inside the cutoff) but twice the set-up; all 8 in every lane, with the
// candidates over the lanes, cost 600 -> 780 us in register moves.  731 us for
// the per-atom kernel, 524 us here (virial on).
//
// Periodic images: an image shift m L is applied where the subtraction is
// exact.  A segment near the upper face, whose neighbours include images
// m = +1, is moved down by L together with its zero-image candidates, so that
// those images stay in place; L is the unevaluated sum Lhi + Llo.
//
// Virial: zero-image pairs through -sum_i c_i F0_i (x) x_i (each is met from
// both atoms with opposite separations, as in the per-atom kernel); pairs of
// other images form their own list and add d (x) d one by one.
//
// Lorentz-Berthelot (LB): records carry sigma, lbw sqrt(2 eps); C_ij =
// lbw_i lbw_j ((sigma_i + sigma_j)/2)^6.
#include <algorithm>
#include <climits>
#include <cmath>
#include <type_traits>

#include "mls6_device.cuh"

namespace mls6 {

struct TileArgs {
  float L[3], Llo[3];  // box length as an unevaluated sum
  float w[3], inv_w[3];
  int nc[3], R[3];
  float a2, ia2, iam;  // a^2, a^-2, 1 / (a + margin)
  float margin;        // absolute slack of the trimming (covers rounding of x, x/w)
  float se, sf;        // a^-6 and 6 a^-8: scales of the sums (lengths in units of a)
};

constexpr int kTileAtoms = 8;
constexpr int kTileWarps = 4;
constexpr int kTileBlocks = 6;  // per SM: 80 registers a thread
constexpr int kTileCap = 384;   // candidates of a list (298 on average at a = 3, density 0.85)
constexpr int kTileRuns = 3 * 25;
constexpr float kTileFar = 1e10f;  // an absent atom or candidate: always outside the cutoff

// ---------------------------------------------------- packed pairs of floats

using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pk(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void upk(f32x2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ float half_sum(f32x2 v) {
  float a, b;
  upk(v, a, b);
  return a + b;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ float rcp_ftz(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float is_zero(float x) {  // 1 if x == 0, else 0
  float r;
  asm("set.eq.f32.f32 %0, %1, 0f00000000;" : "=f"(r) : "f"(x));
  return r;
}

// Sums of one atom of the lane, over the lane's candidates (two halves).
struct TileSum {
  f32x2 e, x, y, z;
};

// Two candidates (packed) against one atom at (-nx, -ny, -nz).  With
// s = (r/a)^2 (1 outside the cutoff), is = 1/s, v = s^3, u = v^2:
//   a^6 g_0           = is^3 - 15/8 + u (5/4 - 3/8 u)
//   -a^8 g_0'/(6 r)   = is^4 - s^5 (5/2 - 3/2 u)
// both 0 at s = 1.  Sums: e += C a^6 g_0, (x, y, z) += C (-a^8 g_0'/6r) d;
// W also w += c_i C (-a^8 g_0'/6r) d (x) d.
template <bool LB, bool W>
__device__ __forceinline__ void tile_pair(TileSum& S, f32x2 (&w)[6], f32x2 qx, f32x2 qy, f32x2 qz,
                                          f32x2 qc, f32x2 qw, f32x2 nx, f32x2 ny, f32x2 nz,
                                          f32x2 ci, f32x2 ia2) {
  const f32x2 dx = add2(qx, nx), dy = add2(qy, ny), dz = add2(qz, nz);
  float s0, s1;
  upk(mul2(fma2(dz, dz, fma2(dy, dy, mul2(dx, dx))), ia2), s0, s1);
  s0 = fminf(s0, 1.0f);
  s1 = fminf(s1, 1.0f);
  const f32x2 s = add2(pk(s0, s1), pk(is_zero(s0), is_zero(s1)));
  upk(s, s0, s1);
  const f32x2 is = pk(rcp_ftz(s0), rcp_ftz(s1));
  const f32x2 s2 = mul2(s, s), v = mul2(s2, s), u = mul2(v, v), s5 = mul2(s2, v);
  const f32x2 i2 = mul2(is, is), i4 = mul2(i2, i2);
  const f32x2 P =
      fma2(u, fma2(u, pk(-0.375f, -0.375f), pk(1.25f, 1.25f)), pk(-1.875f, -1.875f));
  const f32x2 g0 = fma2(i2, is, P);
  const f32x2 gp = fma2(s5, fma2(u, pk(1.5f, 1.5f), pk(-2.5f, -2.5f)), i4);
  f32x2 c = qc;
  if (LB) {  // lbw_j (sigma_i + sigma_j)^6; the factor lbw_i / 64 comes with the scales
    const f32x2 sg = add2(qc, ci), sg2 = mul2(sg, sg), sg3 = mul2(sg2, sg);
    c = mul2(qw, mul2(sg3, sg3));
  }
  S.e = fma2(c, g0, S.e);
  const f32x2 cg = mul2(c, gp);
  S.x = fma2(cg, dx, S.x);
  S.y = fma2(cg, dy, S.y);
  S.z = fma2(cg, dz, S.z);
  if (W) {
    const f32x2 cv = mul2(cg, ci);
    const f32x2 cx = mul2(cv, dx), cy = mul2(cv, dy), cz = mul2(cv, dz);
    w[0] = fma2(cx, dx, w[0]);
    w[1] = fma2(cy, dy, w[1]);
    w[2] = fma2(cz, dz, w[2]);
    w[3] = fma2(cx, dy, w[3]);
    w[4] = fma2(cx, dz, w[4]);
    w[5] = fma2(cy, dz, w[5]);
  }
}

// Shared memory of one warp.  The list is read 16 bytes at a time.
template <bool LB> struct TileShared {
  __align__(16) float x[kTileCap];  // listed candidates
  float y[kTileCap], z[kTileCap], c[kTileCap], w[LB ? kTileCap : 4];
  int run_j[2][kTileRuns];  // runs of the zero image / of other images: first record,
  int run_n[2][kTileRuns];  // length,
  int run_m[kTileRuns];     // image
};
static_assert(kTileCap % 64 == 0 && sizeof(TileShared<true>) % 16 == 0 &&
                  sizeof(TileShared<false>) % 16 == 0,
              "the list's coordinates start at 16-byte boundaries");

// The listed candidates (n of them, filled up to a multiple of 32) against
// the lane's two atoms; at: the atom's frame position and coefficient.
template <bool LB, bool W>
__device__ __forceinline__ void tile_eval(const TileShared<LB>& M, int n, int js, const float4 (&at)[2],
                                          f32x2 ia2, TileSum (&S)[2], f32x2 (&w)[6]) {
  const f32x2 nx0 = pk(-at[0].x, -at[0].x), ny0 = pk(-at[0].y, -at[0].y),
              nz0 = pk(-at[0].z, -at[0].z), c0 = pk(at[0].w, at[0].w);
  const f32x2 nx1 = pk(-at[1].x, -at[1].x), ny1 = pk(-at[1].y, -at[1].y),
              nz1 = pk(-at[1].z, -at[1].z), c1 = pk(at[1].w, at[1].w);
#pragma unroll 1
  for (int u = 4 * js; u < n; u += 32) {
    const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(M.x + u);
    const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(M.y + u);
    const ulonglong2 z = *reinterpret_cast<const ulonglong2*>(M.z + u);
    const ulonglong2 c = *reinterpret_cast<const ulonglong2*>(M.c + u);
    ulonglong2 lw = c;
    if (LB) lw = *reinterpret_cast<const ulonglong2*>(M.w + u);
    tile_pair<LB, W>(S[0], w, x.x, y.x, z.x, c.x, lw.x, nx0, ny0, nz0, c0, ia2);
    tile_pair<LB, W>(S[1], w, x.x, y.x, z.x, c.x, lw.x, nx1, ny1, nz1, c1, ia2);
    tile_pair<LB, W>(S[0], w, x.y, y.y, z.y, c.y, lw.y, nx0, ny0, nz0, c0, ia2);
    tile_pair<LB, W>(S[1], w, x.y, y.y, z.y, c.y, lw.y, nx1, ny1, nz1, c1, ia2);
  }
}

// i = m n + iw with 0 <= iw < n: the cell iw and periodic image m of an
// unwrapped cell index (within one period of the box unless the box is
// thinner than the neighbour range).
__device__ __forceinline__ void tile_wrap(int i, int n, int& iw, int& m) {
  m = i < 0 ? -1 : (i >= n ? 1 : 0);
  iw = i - m * n;
  while (iw < 0) {
    iw += n;
    --m;
  }
  while (iw >= n) {
    iw -= n;
    ++m;
  }
}

// Least and largest over the warp of values >= 0 (their bits order like
// unsigned integers; + 0 turns a negative zero into zero).
__device__ __forceinline__ float warp_min(float v) {
  return __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(v + 0.f)));
}
__device__ __forceinline__ float warp_max(float v) {
  return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v + 0.f)));
}
// 1 << n, 0 for n outside 0..31 (shl clamps the amount)
__device__ __forceinline__ unsigned bit_at(int n) {
  unsigned r;
  asm("shl.b32 %0, 1, %1;" : "=r"(r) : "r"(n));
  return r;
}

template <bool VIR, bool LB>
__global__ void __launch_bounds__(kTileWarps * 32, kTileBlocks) k_pair_tile(
    const float4* __restrict__ sp, const int* __restrict__ start, int N, TileArgs g,
    float* __restrict__ e0, float* __restrict__ floc, double* __restrict__ wpart,
    const float* __restrict__ lbw) {
  constexpr unsigned kAll = 0xffffffffu;
  __shared__ TileShared<LB> shm[kTileWarps];
  __shared__ float wsum[kTileWarps][6];
  __shared__ int ended;  // warps of the block that have written their virial sums
  if (VIR) {
    if (threadIdx.x == 0) ended = 0;
    __syncthreads();
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  TileShared<LB>& M = shm[wid];
  const unsigned below = (1u << lane) - 1u, upto = below | (1u << lane);
  const long warp = (long)blockIdx.x * kTileWarps + wid;
  const long first_atom = warp * kTileAtoms;
  const int gi = lane & 7;                // atom held by this lane
  const int ig = lane & 3, js = lane >> 2;  // evaluation: atoms 2 ig, 2 ig + 1; candidate group
  const int oa = 2 * ig + (js >> 2), oq = js & 3;  // the sum this lane ends up with: atom, e x y z
  float4 pi = make_float4(0.f, 0.f, 0.f, 0.f);
  int cy = 0, cz = 0, rid = INT_MAX;
  if (first_atom + gi < N) {
    pi = sp[first_atom + gi];
    cy = min(max((int)(pi.y * g.inv_w[1]), 0), g.nc[1] - 1);
    cz = min(max((int)(pi.z * g.inv_w[2]), 0), g.nc[2] - 1);
    rid = cy + g.nc[1] * cz;
  }
  float tot = 0.f;                               // sum oq of atom oa
  float w6[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // 2 x virial, in scaled units
#pragma unroll 1
  for (int s = 0; s < kTileAtoms;) {
    const int rs = __shfl_sync(kAll, rid, s);
    if (rs == INT_MAX) break;  // the remaining atoms are past N
    const unsigned seg = __ballot_sync(kAll, lane < kTileAtoms && rid == rs);
    const bool act = (seg >> gi) & 1u;
    // bounding box of the segment
    const float xmn = warp_min(act ? pi.x : INFINITY), xmx = warp_max(act ? pi.x : 0.f);
    const float ymn = warp_min(act ? pi.y : INFINITY), ymx = warp_max(act ? pi.y : 0.f);
    const float zmn = warp_min(act ? pi.z : INFINITY), zmx = warp_max(act ? pi.z : 0.f);
    // 1. lane t: neighbour row t; at most one run of the zero image and
    //    three in all (the range spans at most 2 nc[0] - 1 cells)
    int n0 = 0, n1 = 0;  // runs of the zero image, of other images
    unsigned sides = 0;  // images present: bit d below, bit 4 + d above
    {
      const int ny = 2 * g.R[1] + 1, nrows = (2 * g.R[2] + 1) * ny;
      const int cxmn = min(max((int)(xmn * g.inv_w[0]), 0), g.nc[0] - 1);
      const int cxmx = min(max((int)(xmx * g.inv_w[0]), 0), g.nc[0] - 1);
      const int scy = __shfl_sync(kAll, cy, s), scz = __shfl_sync(kAll, cz, s);
      int xa = 1, xh = 0, ix = 0, mx = 0, row = 0, myz = 0, out = 0;
      if (lane < nrows) {
        const int dz = lane / ny - g.R[2], dy = lane % ny - g.R[1];
        const int z = scz + dz, y = scy + dy;
        int iz, iy, mz, my;
        tile_wrap(z, g.nc[2], iz, mz);
        tile_wrap(y, g.nc[1], iy, my);
        const float ylo = (float)y * g.w[1], zlo = (float)z * g.w[2];
        const float dyl = fmaxf(0.f, fmaxf(ylo - ymx, ymn - (ylo + g.w[1])) - g.margin);
        const float dzl = fmaxf(0.f, fmaxf(zlo - zmx, zmn - (zlo + g.w[2])) - g.margin);
        const float d2 = dyl * dyl + dzl * dzl;
        if (d2 < g.a2) {
          const float rx = sqrtf(g.a2 - d2) + g.margin;
          xa = max(cxmn - g.R[0], (int)floorf((xmn - rx) * g.inv_w[0]));
          xh = min(cxmx + g.R[0], (int)floorf((xmx + rx) * g.inv_w[0]));
          row = g.nc[0] * (iy + g.nc[1] * iz);
          tile_wrap(xa, g.nc[0], ix, mx);
          myz = ((my + 8) << 4) | ((mz + 8) << 8);
          out = my | mz;
          sides = (my < 0 ? 2u : 0u) | (my > 0 ? 32u : 0u) | (mz < 0 ? 4u : 0u) |
                  (mz > 0 ? 64u : 0u);
        }
      }
#pragma unroll 1
      while (__any_sync(kAll, xa <= xh)) {  // run after run of each row (one, away from the faces)
        int j = 0, n = 0;
        const bool zero = (mx | out) == 0;
        const int img = (mx + 8) | myz;
        if (xa <= xh) {
          const int xb = min(xh, xa + (g.nc[0] - 1 - ix));
          j = start[row + ix];
          n = start[row + ix + (xb - xa) + 1] - j;
          sides |= (mx < 0 ? 1u : 0u) | (mx > 0 ? 16u : 0u);
          xa = xb + 1;
          ix = 0;
          ++mx;
        }
        const unsigned m0 = __ballot_sync(kAll, n > 0 && zero);
        const unsigned m1 = __ballot_sync(kAll, n > 0 && !zero);
        if (n > 0) {
          const int t = zero ? n0 + __popc(m0 & below) : n1 + __popc(m1 & below);
          M.run_j[zero ? 0 : 1][t] = j;
          M.run_n[zero ? 0 : 1][t] = n;
          if (!zero) M.run_m[t] = img;
        }
        n0 += __popc(m0);
        n1 += __popc(m1);
      }
      sides = __reduce_or_sync(kAll, sides);
    }
    // frame: moved down by L along an axis with images above and none below
    const float frx = (sides & 0x11u) == 0x10u ? -1.f : 0.f;
    const float fry = (sides & 0x22u) == 0x20u ? -1.f : 0.f;
    const float frz = (sides & 0x44u) == 0x40u ? -1.f : 0.f;
    const float fx = frx * g.L[0], fy = fry * g.L[1], fz = frz * g.L[2];
    float4 at[2];  // the lane's two atoms in the frame
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int src = 2 * ig + k;
      const bool in = (seg >> src) & 1u;
      const float x = __shfl_sync(kAll, pi.x, src), y = __shfl_sync(kAll, pi.y, src);
      const float z = __shfl_sync(kAll, pi.z, src), c = __shfl_sync(kAll, pi.w, src);
      at[k] = make_float4(in ? x + fx : -kTileFar, in ? y + fy : -kTileFar,
                          in ? z + fz : -kTileFar, c);
    }
    const float bx = 0.5f * (xmn + xmx) + fx, by = 0.5f * (ymn + ymx) + fy,
                bz = 0.5f * (zmn + zmx) + fz;
    const float ex = -0.5f * (xmx - xmn) * g.iam, ey = -0.5f * (ymx - ymn) * g.iam,
                ez = -0.5f * (zmx - zmn) * g.iam;
    TileSum S[2];
    f32x2 w2[6] = {0, 0, 0, 0, 0, 0};
    S[0].e = S[0].x = S[0].y = S[0].z = 0;
    S[1] = S[0];
    int cnt = 0;  // candidates in the list
    __syncwarp();
    // the zero image, then the others
#pragma unroll 1
    for (int pass = n0 > 0 ? 0 : 1; pass < (n1 > 0 ? 2 : 1); ++pass) {
      const int nr = pass ? n1 : n0;
      const bool last_pass = pass == 1 || n1 == 0;
#pragma unroll 1
      for (int tg = 0; tg < nr; tg += 32) {
        // lane p: run tg + p and its place in the stream of these runs
        const bool mine = tg + lane < nr;
        const int n = mine ? M.run_n[pass][tg + lane] : 0;
        int inc = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(kAll, inc, o);
          if (lane >= o) inc += v;
        }
        const int total = __shfl_sync(kAll, inc, 31);
        int rel = mine ? inc - n : INT_MAX / 2;  // the run's first candidate, from the window's
        const int base = mine ? M.run_j[pass][tg + lane] - (inc - n) : 0;
        const int img = mine && pass ? M.run_m[tg + lane] : 0;
        int begun = -1;  // runs begun before the window, minus 1
        // 2. windows of 64 candidates: each lane's run from the bits where
        //    runs begin; the two loads in flight together
        auto window = [&](int k, auto framed_c) {
          constexpr bool FR = decltype(framed_c)::value;
          float4 q[2];
          float lw[2] = {0.f, 0.f};
          int im[2] = {0x888, 0x888};
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            const unsigned heads = __reduce_or_sync(kAll, bit_at(rel));
            rel -= 32;
            const int t = begun + __popc(heads & upto);
            begun += __popc(heads);
            const int at_k = k + 32 * v + lane;
            const int j = __shfl_sync(kAll, base, t) + at_k;
            if (FR && pass) im[v] = __shfl_sync(kAll, img, t);
            // past the end: any record, moved out of reach
            const int jc = min(j, N - 1);
            q[v] = sp[jc];
            if (LB) lw[v] = lbw[jc];
            q[v].x = at_k < total ? q[v].x : kTileFar;
          }
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            if (FR) {
              const float mx = (float)((im[v] & 15) - 8), my = (float)(((im[v] >> 4) & 15) - 8),
                          mz = (float)(((im[v] >> 8) & 15) - 8);
              q[v].x = (q[v].x + (mx + frx) * g.L[0]) + mx * g.Llo[0];
              q[v].y = (q[v].y + (my + fry) * g.L[1]) + my * g.Llo[1];
              q[v].z = (q[v].z + (mz + frz) * g.L[2]) + mz * g.Llo[2];
            }
            // distance from the box in units of the reach, each axis clamped to 0..1
            const float dx = __saturatef(fmaf(fabsf(q[v].x - bx), g.iam, ex));
            const float dy = __saturatef(fmaf(fabsf(q[v].y - by), g.iam, ey));
            const float dz = __saturatef(fmaf(fabsf(q[v].z - bz), g.iam, ez));
            const bool hit = dx * dx + dy * dy + dz * dz < 1.0f;
            const unsigned m = __ballot_sync(kAll, hit);
            if (hit) {
              const int t = cnt + __popc(m & below);
              M.x[t] = q[v].x;
              M.y[t] = q[v].y;
              M.z[t] = q[v].z;
              M.c[t] = q[v].w;
              if (LB) M.w[t] = lw[v];
            }
            cnt += __popc(m);
          }
        };
        int k = 0;
#pragma unroll 1
        do {
          // as many windows as the list has room for
          const int end = min(total, k + (kTileCap - cnt) / 64 * 64);
          if (sides == 0) {
#pragma unroll 1
            for (; k < end; k += 64) window(k, std::false_type{});
          } else {
#pragma unroll 1
            for (; k < end; k += 64) window(k, std::true_type{});
          }
          // 3. the list, when it is full or the runs end
          if (cnt > kTileCap - 64 || (k >= total && tg + 32 >= nr && (VIR || last_pass))) {
            const int fill = (cnt + 31) & ~31;
            if (cnt + lane < fill) {
              M.x[cnt + lane] = kTileFar;
              M.y[cnt + lane] = kTileFar;
              M.z[cnt + lane] = kTileFar;
              M.c[cnt + lane] = 0.f;
              if (LB) M.w[cnt + lane] = 0.f;
            }
            __syncwarp();
            const f32x2 ia2 = pk(g.ia2, g.ia2);
            if (VIR && pass)
              tile_eval<LB, VIR>(M, fill, js, at, ia2, S, w2);
            else
              tile_eval<LB, false>(M, fill, js, at, ia2, S, w2);
            __syncwarp();
            cnt = 0;
          }
        } while (k < total);
      }
      // 4. sums over the candidate groups: lane 4 js + ig returns sum js & 3 of atom 2 ig + js / 4
      if (VIR || last_pass) {
        float v[8];
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          v[4 * a + 0] = half_sum(S[a].e);
          v[4 * a + 1] = half_sum(S[a].x);
          v[4 * a + 2] = half_sum(S[a].y);
          v[4 * a + 3] = half_sum(S[a].z);
        }
#pragma unroll
        for (int h = 4; h > 0; h >>= 1) {
          const bool up = js & h;
#pragma unroll
          for (int t = 0; t < h; ++t) {
            const float keep = up ? v[t + h] : v[t], send = up ? v[t] : v[t + h];
            v[t] = keep + __shfl_xor_sync(kAll, send, 4 * h);
          }
        }
        tot += v[0];
        if (VIR) {
          S[0].e = S[0].x = S[0].y = S[0].z = 0;
          S[1] = S[0];
          if (pass == 0) {  // -2 c_i F0_i (x) x_i
            const float x = __shfl_sync(kAll, pi.x, oa), y = __shfl_sync(kAll, pi.y, oa);
            const float z = __shfl_sync(kAll, pi.z, oa), c = __shfl_sync(kAll, pi.w, oa);
            const float f = -2.f * c * v[0];
            if (oq == 1) {
              w6[0] += f * x;
              w6[3] += 0.5f * f * y;
              w6[4] += 0.5f * f * z;
            } else if (oq == 2) {
              w6[1] += f * y;
              w6[3] += 0.5f * f * x;
              w6[5] += 0.5f * f * z;
            } else if (oq == 3) {
              w6[2] += f * z;
              w6[4] += 0.5f * f * x;
              w6[5] += 0.5f * f * y;
            }
          }
        }
      }
    }
    if (VIR && n1 > 0)
#pragma unroll
      for (int c = 0; c < 6; ++c) w6[c] += half_sum(w2[c]);
    __syncwarp();  // the next segment rewrites the tables
    s += __popc(seg);
  }
  // F_i = -c_i sum c_j g_0'/r d = +c_i 6 a^-8 (x, y, z)
  const float c = __shfl_sync(kAll, pi.w, oa);
  if (first_atom + oa < N) {
    const size_t i = (size_t)(first_atom + oa);
    const float ci = LB ? lbw[i] * (1.0f / 64.0f) : c;
    if (oq == 0)
      e0[i] = (LB ? ci * g.se : g.se) * tot;
    else
      floc[3 * i + oq - 1] = ci * g.sf * tot;
  }
  if (VIR) {
    // one record per block, 1/2 sum c_i c_j g_0'/r d (x) d with g_0'/r = -6 a^-8 (...): the
    // warp that ends last adds the warps' sums in their order (no warp waits)
#pragma unroll
    for (int k = 0; k < 6; ++k)
      for (int o = 16; o > 0; o >>= 1) w6[k] += __shfl_down_sync(kAll, w6[k], o);
    bool last = false;
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < 6; ++k) wsum[wid][k] = w6[k];
      __threadfence_block();
      last = atomicAdd(&ended, 1) == kTileWarps - 1;
      __threadfence_block();
    }
    if (__shfl_sync(kAll, (int)last, 0) && lane < 6) {
      double w = 0.0;
#pragma unroll
      for (int v = 0; v < kTileWarps; ++v) w += (double)*(volatile float*)&wsum[v][lane];
      wpart[6 * (size_t)blockIdx.x + lane] = -0.5 * (double)g.sf * w;
    }
  }
}

// The tile form applies where a row of cells meets at most three periodic
// images and the neighbour rows fit in a warp (as for the warp and queue
// forms), in FP32 and mixed plans with the smoothing function of Eq. (gamma).
bool pair_tile_ok(const Plan* p) { return p->prec != MLS6_FP64 && pair_cluster_ok(p); }

int launch_pair_tile(Plan* p, bool vir, bool lb, cudaStream_t st) {
  const int N = (int)p->N;
  const long nb = pair_blocks(p, kPairTile);
  if (nb == 0) return 0;
  TileArgs g;
  for (int d = 0; d < 3; ++d) {
    g.L[d] = (float)p->L[d];
    g.Llo[d] = (float)(p->L[d] - (double)g.L[d]);
    g.w[d] = (float)p->cg.w[d];
    g.inv_w[d] = (float)p->cg.inv_w[d];
    g.nc[d] = p->cg.nc[d];
    g.R[d] = p->cg.R[d];
  }
  // slack: 1e-3 of a cell plus 16 rounding units of the largest coordinate
  const double wmin = std::min(p->cg.w[0], std::min(p->cg.w[1], p->cg.w[2]));
  const double lmax = std::max(p->L[0], std::max(p->L[1], p->L[2]));
  const double margin = 1e-3 * wmin + 16.0 * 6.0e-8 * lmax;
  g.margin = (float)margin;
  g.a2 = (float)(p->a * p->a);
  g.iam = (float)(1.0 / (p->a + margin));
  g.ia2 = (float)(1.0 / (p->a * p->a));
  g.se = (float)std::pow(p->a, -6.0);
  g.sf = (float)(6.0 * std::pow(p->a, -8.0));
  auto k = lb ? k_pair_tile<false, true> : vir ? k_pair_tile<true, false>
                                               : k_pair_tile<false, false>;
  k<<<nb, kTileWarps * 32, 0, st>>>((const float4*)p->d_sorted, p->d_cell_start, N, g,
                                    (float*)p->d_e0, (float*)p->d_floc,
                                    p->d_wpart + 6 * p->wpart_pair,
                                    lb ? (const float*)p->d_lbw : nullptr);
  return 1;
}

}  // namespace mls6
