// Learned force correction for a coarse grid (no counterpart in the paper):
// a small network reads, for each atom, the level-1 total potential of a
// coarse multilevel-summation evaluation around the atom and predicts the
// force residual to a finer evaluation; the correction is c_i * s * y_i.
//
//   features   e^{1,tot} and its gradient interpolated (Eq. interpolation,
//              the method's own basis) at x_i + h d for d in {-1,0,1}^3, and
//              sin / cos of 2 pi times the fractional grid coordinate of x_i:
//              114 values, zero-padded to 128, normalised per feature
//              (shift, scale), stored as BF16 (or FP32) rows in input order
//   network    128 -> 64 -> 64 -> 64 -> 8 (outputs 0..2 used), tanh hidden
//              layers; BF16 weights and activations on the tensor cores
//              (mma.m16n8k16, FP32 accumulation); 16 atoms per tile, the
//              accumulator tiles of a layer are repacked in registers as the
//              A operand of the next
//   training   one kernel per batch: forward, BF16 tensor-core backward pass
//              and weight gradients of a tile of atoms held in shared memory
//              (k_mlp_train); per-block partials summed in a fixed order
//              (results reproducible bit for bit); Adam update of FP32 master
//              weights, BF16 fragments repacked after every step
#include <cuda_bf16.h>
#include <stddef.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "mls6_device.cuh"

namespace mls6 {

#define CK(x)                                    \
  do {                                           \
    cudaError_t e_ = (x);                        \
    if (e_ != cudaSuccess) return MLS6_ERR_CUDA; \
  } while (0)


constexpr int kNF = 128;                        // feature row (114 used)
constexpr int kH = 64;                          // hidden width
constexpr int kNO = 8;                          // output row (3 used)
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kNF * kH;
constexpr int kOffW2 = kOffB1 + kH, kOffB2 = kOffW2 + kH * kH;
constexpr int kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH * kH;
constexpr int kOffW4 = kOffB3 + kH, kOffB4 = kOffW4 + kH * kNO;
constexpr int kNPar = kOffB4 + kNO;             // 17096
// packed B fragments (uint2 per lane): layer 1 8x8 tiles, layers 2-3 4x8, layer 4 4x1
constexpr int kPk1 = 0, kPk2 = kPk1 + 8 * 8 * 32, kPk3 = kPk2 + 4 * 8 * 32,
              kPk4 = kPk3 + 4 * 8 * 32, kPkN = kPk4 + 4 * 1 * 32;
// transposed weights for the backward pass (B[k][n] = W[n][k]): W4^T one
// k-step (K = 8 padded to 16) x 8 tiles, W3^T and W2^T 4 x 8
constexpr int kPkT4 = kPkN, kPkT3 = kPkT4 + 1 * 8 * 32, kPkT2 = kPkT3 + 4 * 8 * 32,
              kPkAll = kPkT2 + 4 * 8 * 32;

struct Mlp {
  float* d_par = nullptr;   // FP32 master weights
  float* d_m = nullptr;     // Adam moments
  float* d_v = nullptr;
  uint2* d_pack = nullptr;  // BF16 B fragments
  float* d_norm = nullptr;  // shift[128], scale[128]
  float out_scale = 1.0f;
  long step = 0;
  cudaStream_t stream = nullptr;
  // work buffers (grown on demand)
  long cap = 0;
  __nv_bfloat16* d_X = nullptr;   // features for mls6_mlp_apply
  float* d_part = nullptr;        // kTGrid x kNPar partial gradients
  double* d_lpart = nullptr;      // loss partials, one per block of k_mlp_train
  float* d_grad = nullptr;        // kNPar
  double* d_loss = nullptr;
};

__device__ __forceinline__ float tanh_fast(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// ------------------------------------------------------------- features

// One thread per (atom, dx): the 9 offsets (dy, dz) of one dx.  Separable: per
// z plane of the 6 x 6 x 6 nodes around the atom an x pass over the 6 rows, a y
// pass for the 3 dy, then the z weights of the dz that the plane belongs to
// (648 multiply-adds a thread; one thread per dz repeats the x and y passes of
// the planes that neighbouring dz share, 1,152).  The block's nodes come from
// shared memory where their box fits (a warp's gathers touched 4 to 8 lines
// each), from global memory otherwise.  A block (3 x kFA threads) assembles
// the rows of kFA atoms in shared memory, on top of the node box, and writes
// each row with 16-byte stores (a row per atom in input order, or in sorted
// order when sorted_out is set).  What
// bounds it: the latency of those reads and sums against 21 warps per SM (four
// blocks, 80 registers, of which 450 bytes of running sums spill): 121 -> 74 us
// at 262,144 atoms (159 registers, no spills, two blocks: 96).
constexpr int kFA = 64;

template <typename T, bool F32>
__global__ void __launch_bounds__(3 * kFA, sizeof(T) == 8 ? 1 : 4) k_features(
    const Vec4<T>* __restrict__ sp, const int* __restrict__ sidx, int N, const T* __restrict__ E,
    int n0, int n1, int n2, T ih0, T ih1, T ih2, const float* __restrict__ norm,
    void* __restrict__ out, int sorted_out) {
  // rows are padded by 16 bytes: those of eight atoms start in distinct banks
  constexpr int kRow = (F32 ? 4 : 2) * kNF + 16;
  constexpr int kBytes = kFA * kRow > kNodeBoxBytes ? kFA * kRow : kNodeBoxBytes;
  __shared__ __align__(16) unsigned char smem[kBytes];
  T* box = reinterpret_cast<T*>(smem);
  const int la = threadIdx.x / 3, dx = (int)(threadIdx.x % 3);
  const int i = blockIdx.x * kFA + la;
  const bool valid = i < N;
  const Vec4<T> p = valid ? sp[i] : Vec4<T>{T(0), T(0), T(0), T(0)};
  const T u0 = p.x * ih0, u1 = p.y * ih1, u2 = p.z * ih2;
  const T f0 = floor(u0), f1 = floor(u1), f2 = floor(u2);
  const int b0 = (int)f0, b1 = (int)f1, b2 = (int)f2;
  const NodeBox B =
      block_node_box<2, 3>(valid, b0, b1, b2, n0, n1, n2, kNodeBoxBytes / (int)sizeof(T));
  if (B.in) load_node_box(box, E, B, n0, n1, n2);
  T e[9], gx[9], gy[9], gz[9];  // offset k = dy + 3 dz
#pragma unroll
  for (int k = 0; k < 9; ++k) e[k] = gx[k] = gy[k] = gz[k] = T(0);
  if (valid) {
    T wx[4], dwx[4], wy[4], dwy[4], wz[4], dwz[4];
    phi4(u0 - f0, wx, dwx);
    phi4(u1 - f1, wy, dwy);
    phi4(u2 - f2, wz, dwz);
    auto sums = [&](auto node) {
#pragma unroll
      for (int c = 0; c < 6; ++c) {  // plane z = b2 - 2 + c
        T ax[6], bx[6];
#pragma unroll
        for (int yy = 0; yy < 6; ++yy) {
          T s = 0, ds = 0;
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            const T v = node(c, yy, a);
            s += wx[a] * v;
            ds += dwx[a] * v;
          }
          ax[yy] = s;
          bx[yy] = ds;
        }
#pragma unroll
        for (int dy = 0; dy < 3; ++dy) {
          T aa = 0, ab = 0, ba = 0;
#pragma unroll
          for (int bb = 0; bb < 4; ++bb) {
            aa += wy[bb] * ax[dy + bb];
            ab += dwy[bb] * ax[dy + bb];
            ba += wy[bb] * bx[dy + bb];
          }
#pragma unroll
          for (int dz = 0; dz < 3; ++dz) {
            const int m = c - dz;  // the plane's place in the support of offset dz
            if (m < 0 || m > 3) continue;
            const int k = dy + 3 * dz;
            e[k] += wz[m] * aa;
            gz[k] += dwz[m] * aa;
            gy[k] += wz[m] * ab;
            gx[k] += wz[m] * ba;
          }
        }
      }
    };
    if (B.in) {
      const T* at = box + (b0 - 2 - B.lo0 + dx) +
                    B.e0 * ((b1 - 2 - B.lo1) + B.e1 * (b2 - 2 - B.lo2));
      const int sy = B.e0, sz = B.e0 * B.e1;
      sums([&](int c, int yy, int a) { return at[c * sz + yy * sy + a]; });
    } else {
      int ix[4], iy[6], iz[6];
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        iy[k] = wrapi(b1 - 2 + k, n1);
        iz[k] = wrapi(b2 - 2 + k, n2);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) ix[k] = wrapi(b0 - 2 + dx + k, n0);
      sums([&](int c, int yy, int a) {
        return E[(long)n0 * (iy[yy] + (long)n1 * iz[c]) + ix[a]];
      });
    }
  }
  __syncthreads();  // the node box is read: its memory takes the rows
  unsigned char* row = smem + la * kRow;
  auto scaled = [&](int j, float v) { return (v - norm[j]) * norm[kNF + j]; };
  auto put2 = [&](int j, float v0, float v1) {  // columns j, j + 1 (j even)
    const float a = scaled(j, v0), b = scaled(j + 1, v1);
    if (F32)
      *reinterpret_cast<float2*>(row + 4 * j) = make_float2(a, b);
    else
      *reinterpret_cast<uint32_t*>(row + 2 * j) = pack_bf16(a, b);
  };
  if (valid) {
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const int j = 4 * (dx + 3 * k);
      const float4 sh = *reinterpret_cast<const float4*>(norm + j);
      const float4 sc = *reinterpret_cast<const float4*>(norm + kNF + j);
      const float v0 = ((float)e[k] - sh.x) * sc.x;
      const float v1 = ((float)(gx[k] * ih0) - sh.y) * sc.y;
      const float v2 = ((float)(gy[k] * ih1) - sh.z) * sc.z;
      const float v3 = ((float)(gz[k] * ih2) - sh.w) * sc.w;
      if (F32)
        *reinterpret_cast<float4*>(row + 4 * j) = make_float4(v0, v1, v2, v3);
      else
        *reinterpret_cast<uint2*>(row + 2 * j) = make_uint2(pack_bf16(v0, v1), pack_bf16(v2, v3));
    }
    const float t = (float)(dx == 0 ? u0 - f0 : dx == 1 ? u1 - f1 : u2 - f2);
    float s, co;
    sincospif(2.0f * t, &s, &co);
    put2(108 + 2 * dx, s, co);
    for (int j = 114 + 2 * dx; j < kNF; j += 6) put2(j, 0.0f, 0.0f);
  }
  __syncthreads();
  // rows out: 16-byte pieces (8 bf16 or 4 floats)
  constexpr int per = F32 ? kNF / 4 : kNF / 8;
  for (int t = threadIdx.x; t < kFA * per; t += blockDim.x) {
    const int a = t / per, ch = t % per;
    const int ii = blockIdx.x * kFA + a;
    if (ii >= N) continue;
    const long r = sorted_out ? ii : sidx[ii];
    reinterpret_cast<uint4*>(out)[r * per + ch] =
        *reinterpret_cast<const uint4*>(smem + a * kRow + 16 * ch);
  }
}

// ----------------------------------------------------------------- network

// B fragment of mma.m16n8k16 for weights W (K x N row-major, row = input):
// lane (g = lane/4, c2 = 2*(lane%4)) holds W[16ks+c2..+1][8nt+g] and
// W[16ks+c2+8..+9][8nt+g].
// Transposed (backward) fragments: B[k][n] = W[n][k] for W = W4, W3, W2
// (row = input n, column = output k); k >= the layer's outputs is zero.
__device__ __forceinline__ float wt_at(const float* W, int NO, int k, int n) {
  return k < NO ? W[n * NO + k] : 0.f;
}

__global__ void k_mlp_pack(const float* __restrict__ par, uint2* __restrict__ pk) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= kPkAll) return;
  if (t >= kPkN) {
    int off, NO, base;
    if (t < kPkT3) {
      off = kOffW4; NO = kNO; base = kPkT4;
    } else if (t < kPkT2) {
      off = kOffW3; NO = kH; base = kPkT3;
    } else {
      off = kOffW2; NO = kH; base = kPkT2;
    }
    const int r = t - base, lane = r & 31, tile = r >> 5;
    const int ks = tile / 8, nt = tile % 8;
    const int g = lane >> 2, c2 = (lane & 3) * 2;
    const int n = 8 * nt + g, k = 16 * ks + c2;
    const float* W = par + off;
    uint2 v;
    v.x = pack_bf16(wt_at(W, NO, k, n), wt_at(W, NO, k + 1, n));
    v.y = pack_bf16(wt_at(W, NO, k + 8, n), wt_at(W, NO, k + 9, n));
    pk[t] = v;
    return;
  }
  int off, NT, NO, base;
  if (t < kPk2) {
    off = kOffW1; NT = 8; NO = kH; base = kPk1;
  } else if (t < kPk3) {
    off = kOffW2; NT = 8; NO = kH; base = kPk2;
  } else if (t < kPk4) {
    off = kOffW3; NT = 8; NO = kH; base = kPk3;
  } else {
    off = kOffW4; NT = 1; NO = kNO; base = kPk4;
  }
  const int r = t - base, lane = r & 31, tile = r >> 5;
  const int ks = tile / NT, nt = tile % NT;
  const int g = lane >> 2, c2 = (lane & 3) * 2;
  const int n = 8 * nt + g, k = 16 * ks + c2;
  const float* W = par + off;
  uint2 v;
  v.x = pack_bf16(W[(k + 0) * NO + n], W[(k + 1) * NO + n]);
  v.y = pack_bf16(W[(k + 8) * NO + n], W[(k + 9) * NO + n]);
  pk[t] = v;
}

// bias + tanh of accumulator tiles (2 per k-step of the next layer), packed
// as the next layer's A fragments: acc[2ks] gives rows g / g+8 at columns
// c2.., acc[2ks+1] the columns c2+8...
__device__ __forceinline__ void next_a(const float (&acc)[8][4], const float* __restrict__ b,
                                       int c2, uint32_t (&A)[4][4]) {
#pragma unroll
  for (int ks = 0; ks < 4; ++ks) {
    const int n0 = 16 * ks + c2, n1 = n0 + 8;
    A[ks][0] = pack_bf16(tanh_fast(acc[2 * ks][0] + b[n0]), tanh_fast(acc[2 * ks][1] + b[n0 + 1]));
    A[ks][1] = pack_bf16(tanh_fast(acc[2 * ks][2] + b[n0]), tanh_fast(acc[2 * ks][3] + b[n0 + 1]));
    A[ks][2] = pack_bf16(tanh_fast(acc[2 * ks + 1][0] + b[n1]),
                         tanh_fast(acc[2 * ks + 1][1] + b[n1 + 1]));
    A[ks][3] = pack_bf16(tanh_fast(acc[2 * ks + 1][2] + b[n1]),
                         tanh_fast(acc[2 * ks + 1][3] + b[n1 + 1]));
  }
}

__device__ __forceinline__ void hidden_layer(const uint32_t (&A)[4][4], const uint2* __restrict__ sw,
                                             int lane, float (&acc)[8][4]) {
#pragma unroll
  for (int nt = 0; nt < 8; ++nt)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[nt][c] = 0.f;
#pragma unroll
  for (int ks = 0; ks < 4; ++ks)
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      const uint2 b = sw[(ks * 8 + nt) * 32 + lane];
      mma16816(acc[nt], A[ks][0], A[ks][1], A[ks][2], A[ks][3], b.x, b.y);
    }
}

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const void* p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a)
               : "memory");
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src, int bytes) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void cp_async4(void* dst, const void* src, int bytes) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(bytes)
               : "memory");
}

// Feature rows in shared memory: the 16-byte piece q of row r lies at piece
// q ^ (r & 7), so that the eight rows of an ldmatrix lie in distinct banks.
__device__ __forceinline__ __nv_bfloat16* x_piece(__nv_bfloat16* x, int r, int q) {
  return x + r * kNF + 8 * (q ^ (r & 7));
}

// A fragment of layer 1: rows row0 .. row0 + 15, k-step ks.
__device__ __forceinline__ void frag_x(uint32_t (&a)[4], __nv_bfloat16* x, int row0, int ks,
                                       int lane) {
  const int j = lane >> 3, r = lane & 7;
  ldsm4(a, x_piece(x, row0 + r + 8 * (j & 1), 2 * ks + (j >> 1)));
}

// Forward pass, 32 rows per warp and step: two 16-row tiles share every weight
// fragment (16 rows per warp read the fragments from shared memory twice as
// often as the tensor cores could use them), and the next 32 rows are copied
// into the warp's other buffer meanwhile.  Either the outputs are stored (Y,
// N x 8), or, with sp given, the rows are the sorted atoms and the correction
// is added to the forces of atom o = sidx[row]: F_o += c_o s y.
// x16: rows start on 16-byte boundaries (else they are copied by words).
// What bounds it: 132 mma and 96 tanh.approx per 16 rows and lane.  262,144
// rows: 50 -> 29 us; with the correction as its last step instead of a kernel
// that reads the outputs back, 64 -> 41.
constexpr int kFwdWarps = 8, kFwdRows = 32;
struct FwdShared {
  __nv_bfloat16 x[kFwdWarps][2][kFwdRows * kNF];
  uint2 w[kPkN];
  float b[3 * kH + kNO];
};
static_assert(sizeof(FwdShared) <= 227 * 1024, "shared memory of one block");

template <typename T>
struct Correction {
  const Vec4<T>* sp;
  const int* sidx;
  T s;
  T* F;
};

template <typename T>
__global__ void __launch_bounds__(32 * kFwdWarps, 1)
    k_mlp_fwd(const __nv_bfloat16* __restrict__ X, long N, int x16, const uint2* __restrict__ pk,
              const float* __restrict__ par, float* __restrict__ Y, Correction<T> C) {
  extern __shared__ __align__(16) unsigned char mlp_smem[];
  FwdShared& S = *reinterpret_cast<FwdShared*>(mlp_smem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, c2 = (lane & 3) * 2;
  auto stage = [&](int st, long tile) {
    __nv_bfloat16* x = S.x[warp][st];
    const long r0 = tile * kFwdRows;
    if (x16) {
#pragma unroll
      for (int t = lane; t < kFwdRows * (kNF / 8); t += 32) {
        const int r = t / (kNF / 8), q = t % (kNF / 8);
        const bool ok = r0 + r < N;
        cp_async16(x_piece(x, r, q), X + (ok ? r0 + r : 0) * kNF + 8 * q, ok ? 16 : 0);
      }
    } else {
      for (int t = lane; t < kFwdRows * (kNF / 2); t += 32) {
        const int r = t / (kNF / 2), q = t % (kNF / 2);
        const bool ok = r0 + r < N;
        cp_async4(x_piece(x, r, q >> 2) + 2 * (q & 3), X + (ok ? r0 + r : 0) * kNF + 2 * q,
                  ok ? 4 : 0);
      }
    }
  };
  const long first = (long)blockIdx.x * kFwdWarps + warp, step = (long)gridDim.x * kFwdWarps;
  if (first * kFwdRows < N) stage(0, first);
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  for (int i = threadIdx.x; i < kPkN; i += blockDim.x) S.w[i] = pk[i];
  for (int i = threadIdx.x; i < kH; i += blockDim.x) {
    S.b[i] = par[kOffB1 + i];
    S.b[kH + i] = par[kOffB2 + i];
    S.b[2 * kH + i] = par[kOffB3 + i];
  }
  if (threadIdx.x < kNO) S.b[3 * kH + threadIdx.x] = par[kOffB4 + threadIdx.x];
  __syncthreads();
  int st = 0;
  for (long tile = first; tile * kFwdRows < N; tile += step, st ^= 1) {
    if ((tile + step) * kFwdRows < N) stage(st ^ 1, tile + step);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncwarp();
    // what the correction needs, ahead of the products that hide its latency
    T cf[4] = {}, fo[4][2] = {};
    T* fp[4] = {};
    if (C.sp && c2 < 3)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const long r = tile * kFwdRows + 16 * (q >> 1) + 8 * (q & 1) + g;
        if (r >= N) continue;
        cf[q] = C.sp[r].w * C.s;
        fp[q] = C.F + 3 * (size_t)C.sidx[r] + c2;
        fo[q][0] = fp[q][0];
        if (c2 == 0) fo[q][1] = fp[q][1];
      }
    float acc[2][8][4];
    uint32_t A[2][4][4];
    auto clear = [&] {
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int nt = 0; nt < 8; ++nt)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[m][nt][c] = 0.f;
    };
    // layer 1: K = 128 (8 k-steps), N = 64 (8 tiles)
    clear();
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
      uint32_t xa[2][4];
      frag_x(xa[0], S.x[warp][st], 0, ks, lane);
      frag_x(xa[1], S.x[warp][st], 16, ks, lane);
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        const uint2 b = S.w[kPk1 + (ks * 8 + nt) * 32 + lane];
#pragma unroll
        for (int m = 0; m < 2; ++m)
          mma16816(acc[m][nt], xa[m][0], xa[m][1], xa[m][2], xa[m][3], b.x, b.y);
      }
    }
    next_a(acc[0], S.b, c2, A[0]);
    next_a(acc[1], S.b, c2, A[1]);
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      const uint2* w = S.w + (l ? kPk3 : kPk2);
      clear();
#pragma unroll
      for (int ks = 0; ks < 4; ++ks)
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
          const uint2 b = w[(ks * 8 + nt) * 32 + lane];
#pragma unroll
          for (int m = 0; m < 2; ++m)
            mma16816(acc[m][nt], A[m][ks][0], A[m][ks][1], A[m][ks][2], A[m][ks][3], b.x, b.y);
        }
      next_a(acc[0], S.b + (l + 1) * kH, c2, A[0]);
      next_a(acc[1], S.b + (l + 1) * kH, c2, A[1]);
    }
    // output layer: N = 8 (one tile)
    float o[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      const uint2 b = S.w[kPk4 + ks * 32 + lane];
#pragma unroll
      for (int m = 0; m < 2; ++m)
        mma16816(o[m], A[m][ks][0], A[m][ks][1], A[m][ks][2], A[m][ks][3], b.x, b.y);
    }
    const float b40 = S.b[3 * kH + c2], b41 = S.b[3 * kH + c2 + 1];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const long r = tile * kFwdRows + 16 * (q >> 1) + 8 * (q & 1) + g;
      const float y0 = o[q >> 1][2 * (q & 1)] + b40, y1 = o[q >> 1][2 * (q & 1) + 1] + b41;
      if (r >= N) continue;
      if (C.sp) {
        if (c2 < 3) {
          fp[q][0] = fo[q][0] + cf[q] * (T)y0;
          if (c2 == 0) fp[q][1] = fo[q][1] + cf[q] * (T)y1;
        }
      } else {
        Y[r * kNO + c2] = y0;
        Y[r * kNO + c2 + 1] = y1;
      }
    }
    __syncwarp();  // the buffer is read: the next step fills it
  }
}

// ---------------------------------------------------------------- training

// Loss and gradient of a batch in one pass over the rows.  A block of 8 warps
// takes `per` consecutive tiles of kTA atoms; per tile
//   - every warp runs the network on its 16 atoms:
//     activations stay in registers as the next layer's A fragments and go to
//     shared memory as rows [atom][unit];
//   - dY = 2 (y - t) / N on outputs 0..2 (BF16), then per layer
//       dZ3 = (dY W4^T) (1 - h3^2),  dZ2 = (dZ3 W3^T) (1 - h2^2),
//       dZ1 = (dZ2 W2^T) (1 - h1^2),
//     each product an mma over the transposed-weight fragments with FP32
//     accumulators, the result packed (BF16) both as the next product's A
//     fragments and into shared memory;
//   - the block adds the tile to its weight gradients,
//       dW1 = X^T dZ1 (128 x 64), dW2 = H1^T dZ2, dW3 = H2^T dZ3 (64 x 64),
//       dW4 = H3^T dY (64 x 8), db = column sums of dZ1, dZ2, dZ3, dY,
//     with the atoms as the K dimension: both operands are read from the rows
//     in shared memory with ldmatrix .trans.  Warp w owns rows 16w.. of dW1,
//     rows 16w.. of dW2 and dW4 (w < 4) or of dW3 (w >= 4); the bias sums are
//     products with an all-ones A (every row of the result is the column
//     sum), taken by warps 0 (b2), 1 (b4), 4 (b1), 5 (b3) from fragments they
//     already hold.
// The features of the next tile are copied (cp.async, 16-byte pieces, rows
// past N zero) while a tile is used.  Partials go to part[block][*] and
// lpart[block]; k_mlp_reduce sums them in block order: results are
// reproducible bit for bit.
// What bounds it: the chain of dependent mma and tanh of a warp (two warps per
// scheduler), not memory: X and T are read once.  Three kernels (forward,
// backward, weight gradients) passed 3 x N x 64 activations and as many
// gradients through memory instead, 93 us at 65,536 atoms against 37.
// 128 atoms per tile: 16 per warp, and 226 KB of rows, two feature stages and
// weight fragments are what one SM holds.
constexpr int kTA = 128, kTGrid = 152;  // atoms per tile, most blocks (partials)
constexpr int kHS = kH + 8;             // row pitch: 8 rows of an ldmatrix in distinct banks

struct TrainShared {
  __nv_bfloat16 x[2][kTA * kNF];  // pieces as in x_piece
  __nv_bfloat16 h[3][kTA * kHS];
  __nv_bfloat16 d[3][kTA * kHS];
  __nv_bfloat16 dy[kTA * kNO];
  uint2 w[kPkAll];
  float b[3 * kH + kNO];
  double loss[8];
};
static_assert(sizeof(TrainShared) <= 227 * 1024, "shared memory of one block");
static_assert(offsetof(TrainShared, h) % 16 == 0 && offsetof(TrainShared, d) % 16 == 0 &&
                  offsetof(TrainShared, dy) % 16 == 0 && offsetof(TrainShared, w) % 16 == 0 &&
                  offsetof(TrainShared, loss) % 8 == 0,
              "alignment of the shared-memory rows");

__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const void* p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a)
               : "memory");
}

__device__ __forceinline__ void ldsm2t(uint32_t (&r)[2], const void* p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n"
               : "=r"(r[0]), "=r"(r[1])
               : "r"(a)
               : "memory");
}

// A fragments of rows 16 m0.. (the activation columns) for k-step ks of a
// tile [atom][column]: matrices (atoms 0-7 / 8-15) x (columns 0-7 / 8-15) in
// the order a0 a1 a2 a3 of the mma.
__device__ __forceinline__ void frag_a(uint32_t (&a)[4], const __nv_bfloat16* t, int ks, int m0,
                                       int lane) {
  const int j = lane >> 3, r = lane & 7;
  ldsm4t(a, t + (16 * ks + r + 8 * (j >> 1)) * kHS + 16 * m0 + 8 * (j & 1));
}

__device__ __forceinline__ void frag_ax(uint32_t (&a)[4], __nv_bfloat16* x, int ks, int m0,
                                        int lane) {
  const int j = lane >> 3, r = lane & 7;
  ldsm4t(a, x_piece(x, 16 * ks + r + 8 * (j >> 1), 2 * m0 + (j & 1)));
}

// B fragments of column tiles nt0, nt0+1 for k-step ks: b[0..1] for nt0,
// b[2..3] for nt0+1.
__device__ __forceinline__ void frag_b2(uint32_t (&b)[4], const __nv_bfloat16* t, int ks, int nt0,
                                        int lane) {
  const int j = lane >> 3, r = lane & 7;
  ldsm4t(b, t + (16 * ks + r + 8 * (j & 1)) * kHS + 8 * (nt0 + (j >> 1)));
}

// Fragments of a warp's 16 rows (g and g + 8 of row0) as rows of a tile; rows
// past the batch (va, vb false) are zero, so that they add nothing.
__device__ __forceinline__ void put_rows(__nv_bfloat16* t, int row0, int g, bool va, bool vb,
                                         int c2, const uint32_t (&A)[4][4]) {
  uint32_t* pa = reinterpret_cast<uint32_t*>(t + (row0 + g) * kHS + c2);
  uint32_t* pb = reinterpret_cast<uint32_t*>(t + (row0 + g + 8) * kHS + c2);
#pragma unroll
  for (int ks = 0; ks < 4; ++ks) {
    pa[8 * ks] = va ? A[ks][0] : 0u;
    pb[8 * ks] = vb ? A[ks][1] : 0u;
    pa[8 * ks + 4] = va ? A[ks][2] : 0u;
    pb[8 * ks + 4] = vb ? A[ks][3] : 0u;
  }
}

__device__ __forceinline__ void get_rows(const __nv_bfloat16* t, int row0, int g, int c2,
                                         uint32_t (&A)[4][4]) {
  const uint32_t* pa = reinterpret_cast<const uint32_t*>(t + (row0 + g) * kHS + c2);
  const uint32_t* pb = reinterpret_cast<const uint32_t*>(t + (row0 + g + 8) * kHS + c2);
#pragma unroll
  for (int ks = 0; ks < 4; ++ks) {
    A[ks][0] = pa[8 * ks];
    A[ks][1] = pb[8 * ks];
    A[ks][2] = pa[8 * ks + 4];
    A[ks][3] = pb[8 * ks + 4];
  }
}

// v (1 - h^2) for two columns, packed.
__device__ __forceinline__ uint32_t act_grad2(float v0, float v1, uint32_t h2) {
  const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(&h2);
  const float h0 = __low2float(h), h1 = __high2float(h);
  return pack_bf16(v0 * (1.f - h0 * h0), v1 * (1.f - h1 * h1));
}

// Column tile nt of acc is half (nt & 1) of k-step nt / 2 of the next product.
__device__ __forceinline__ void act_grad(const float (&acc)[8][4], const uint32_t (&H)[4][4],
                                         uint32_t (&A)[4][4]) {
#pragma unroll
  for (int nt = 0; nt < 8; ++nt) {
    const int ks = nt >> 1, o = (nt & 1) * 2;
    A[ks][o] = act_grad2(acc[nt][0], acc[nt][1], H[ks][o]);
    A[ks][o + 1] = act_grad2(acc[nt][2], acc[nt][3], H[ks][o + 1]);
  }
}

__global__ void __launch_bounds__(256, 1) k_mlp_train(
    const __nv_bfloat16* __restrict__ X, const float* __restrict__ T, long N, long per,
    float inv_n, const uint2* __restrict__ pk, const float* __restrict__ par,
    float* __restrict__ part, double* __restrict__ lpart) {
  extern __shared__ __align__(16) unsigned char mlp_smem[];
  TrainShared& S = *reinterpret_cast<TrainShared*>(mlp_smem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, c2 = (lane & 3) * 2;
  const long ntile = cdiv(N, (long)kTA);
  const long t0 = (long)blockIdx.x * per, t1 = min(ntile, t0 + per);
  auto stage = [&](int st, long tile) {
    for (int t = threadIdx.x; t < kTA * (kNF / 8); t += blockDim.x) {
      const int r = t / (kNF / 8), q = t % (kNF / 8);
      const long i = tile * kTA + r;
      const bool ok = i < N;
      cp_async16(x_piece(S.x[st], r, q), X + (ok ? i : 0) * kNF + 8 * q,
                 ok ? 16 : 0);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  if (t0 < t1) stage(0, t0);
  for (int i = threadIdx.x; i < kPkAll; i += blockDim.x) S.w[i] = pk[i];
  for (int i = threadIdx.x; i < kH; i += blockDim.x) {
    S.b[i] = par[kOffB1 + i];
    S.b[kH + i] = par[kOffB2 + i];
    S.b[2 * kH + i] = par[kOffB3 + i];
  }
  if (threadIdx.x < kNO) S.b[3 * kH + threadIdx.x] = par[kOffB4 + threadIdx.x];

  float a1[8][4], a23[8][4], a4[4], ab[8][4];
#pragma unroll
  for (int n = 0; n < 8; ++n)
#pragma unroll
    for (int c = 0; c < 4; ++c) a1[n][c] = a23[n][c] = ab[n][c] = 0.f;
#pragma unroll
  for (int c = 0; c < 4; ++c) a4[c] = 0.f;
  const uint32_t one = 0x3F803F80u;  // two BF16 ones
  double l = 0.0;

  for (long tile = t0; tile < t1; ++tile) {
    const int st = (int)((tile - t0) & 1);
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();  // stage st filled; the other stage and all rows are free
    if (tile + 1 < t1) stage(st ^ 1, tile + 1);
    const int row0 = 16 * warp;
    const long ra = tile * kTA + row0 + g, rb = ra + 8;
    const bool va = ra < N, vb = rb < N;
    float tg[4];  // targets (ra, c2), (ra, c2 + 1), (rb, c2), (rb, c2 + 1)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = c2 + (q & 1);
      tg[q] = ((q < 2 ? va : vb) && c < 3) ? T[(q < 2 ? ra : rb) * 3 + c] : 0.f;
    }
    // forward
    float acc[8][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[nt][c] = 0.f;
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
      uint32_t xa[4];
      frag_x(xa, S.x[st], row0, ks, lane);
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        const uint2 b = S.w[kPk1 + (ks * 8 + nt) * 32 + lane];
        mma16816(acc[nt], xa[0], xa[1], xa[2], xa[3], b.x, b.y);
      }
    }
    uint32_t A[4][4], H[4][4];
    next_a(acc, S.b, c2, A);
    put_rows(S.h[0], row0, g, va, vb, c2, A);
    hidden_layer(A, S.w + kPk2, lane, acc);
    next_a(acc, S.b + kH, c2, A);
    put_rows(S.h[1], row0, g, va, vb, c2, A);
    hidden_layer(A, S.w + kPk3, lane, acc);
    next_a(acc, S.b + 2 * kH, c2, H);
    put_rows(S.h[2], row0, g, va, vb, c2, H);
    float o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      const uint2 b = S.w[kPk4 + ks * 32 + lane];
      mma16816(o, H[ks][0], H[ks][1], H[ks][2], H[ks][3], b.x, b.y);
    }
    // output gradients and loss
    float dy[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = c2 + (q & 1);
      if ((q < 2 ? va : vb) && c < 3) {
        const float e = o[q] + S.b[3 * kH + c] - tg[q];
        l += (double)e * e;
        dy[q] = 2.f * e * inv_n;
      }
    }
    const uint32_t da = pack_bf16(dy[0], dy[1]), db = pack_bf16(dy[2], dy[3]);
    *reinterpret_cast<uint32_t*>(S.dy + (row0 + g) * kNO + c2) = da;
    *reinterpret_cast<uint32_t*>(S.dy + (row0 + g + 8) * kNO + c2) = db;
    // backward: dY W4^T is one k-step, columns 8..15 of A are zero
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.f;
      const uint2 b = S.w[kPkT4 + nt * 32 + lane];
      mma16816(acc[nt], da, db, 0u, 0u, b.x, b.y);
    }
    act_grad(acc, H, A);
    put_rows(S.d[2], row0, g, va, vb, c2, A);
    hidden_layer(A, S.w + kPkT3, lane, acc);
    get_rows(S.h[1], row0, g, c2, H);  // this thread's own words
    act_grad(acc, H, A);
    put_rows(S.d[1], row0, g, va, vb, c2, A);
    hidden_layer(A, S.w + kPkT2, lane, acc);
    get_rows(S.h[0], row0, g, c2, H);
    act_grad(acc, H, A);
    put_rows(S.d[0], row0, g, va, vb, c2, A);
    __syncthreads();  // the tile's rows are complete

    // weight gradients
    const int l23 = warp < 4 ? 0 : 1;  // dW2 (H1, dZ2) or dW3 (H2, dZ3)
    const int m23 = warp & 3;
#pragma unroll 2
    for (int ks = 0; ks < kTA / 16; ++ks) {
      uint32_t a[4], b[4][4];
      // dW1 rows 16 warp..: X^T dZ1
      frag_ax(a, S.x[st], ks, warp, lane);
#pragma unroll
      for (int q = 0; q < 4; ++q) frag_b2(b[q], S.d[0], ks, 2 * q, lane);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        mma16816(a1[2 * q], a[0], a[1], a[2], a[3], b[q][0], b[q][1]);
        mma16816(a1[2 * q + 1], a[0], a[1], a[2], a[3], b[q][2], b[q][3]);
      }
      if (warp == 4)  // b1: column sums of dZ1
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          mma16816(ab[2 * q], one, one, one, one, b[q][0], b[q][1]);
          mma16816(ab[2 * q + 1], one, one, one, one, b[q][2], b[q][3]);
        }
      // dW2 (warps 0-3) / dW3 (warps 4-7)
      frag_a(a, S.h[l23], ks, m23, lane);
#pragma unroll
      for (int q = 0; q < 4; ++q) frag_b2(b[q], S.d[1 + l23], ks, 2 * q, lane);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        mma16816(a23[2 * q], a[0], a[1], a[2], a[3], b[q][0], b[q][1]);
        mma16816(a23[2 * q + 1], a[0], a[1], a[2], a[3], b[q][2], b[q][3]);
      }
      if (warp == 0 || warp == 5)  // b2 (dZ2) / b3 (dZ3)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          mma16816(ab[2 * q], one, one, one, one, b[q][0], b[q][1]);
          mma16816(ab[2 * q + 1], one, one, one, one, b[q][2], b[q][3]);
        }
      if (warp < 4) {  // dW4 rows 16 warp..: H3^T dY (one column tile)
        uint32_t by[2];
        {
          const int j = (lane >> 3) & 1, r = lane & 7;
          ldsm2t(by, S.dy + (16 * ks + r + 8 * j) * kNO);
        }
        frag_a(a, S.h[2], ks, warp, lane);
        mma16816(a4, a[0], a[1], a[2], a[3], by[0], by[1]);
        if (warp == 1) mma16816(ab[0], one, one, one, one, by[0], by[1]);  // b4
      }
    }
  }

  // partial of this block, parameter order of the master weights
  float* P = part + (long)blockIdx.x * kNPar;
#pragma unroll
  for (int nt = 0; nt < 8; ++nt)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int m = g + 8 * (c >> 1), n = 8 * nt + c2 + (c & 1);
      P[kOffW1 + (16 * warp + m) * kH + n] = a1[nt][c];
      P[(warp < 4 ? kOffW2 : kOffW3) + (16 * (warp & 3) + m) * kH + n] = a23[nt][c];
    }
  if (warp < 4)
#pragma unroll
    for (int c = 0; c < 4; ++c)
      P[kOffW4 + (16 * warp + g + 8 * (c >> 1)) * kNO + c2 + (c & 1)] = a4[c];
  if (g == 0) {  // row 0 of the ones products
    if (warp == 4 || warp == 0 || warp == 5)
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        const int off = warp == 4 ? kOffB1 : (warp == 0 ? kOffB2 : kOffB3);
        P[off + 8 * nt + c2] = ab[nt][0];
        P[off + 8 * nt + c2 + 1] = ab[nt][1];
      }
    if (warp == 1) {
      P[kOffB4 + c2] = ab[0][0];
      P[kOffB4 + c2 + 1] = ab[0][1];
    }
  }
  l = warp_sum(l);
  if (lane == 0) S.loss[warp] = l;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) l += S.loss[w];
    lpart[blockIdx.x] = l;
  }
}

// Fixed-order sums over the blocks' partials: gradient (FP32 out, summed in
// FP64; also to grad_out where given) and the loss.  32 parameters per block;
// thread row s adds the partials s, s + 8, ... and the rows' sums are added in
// order.  One thread per parameter left 85 of the 152 SMs idle, and its block
// 0 added 1,024 loss partials in one chain: 84 us against 13 at 65,536
// atoms.
__global__ void __launch_bounds__(256) k_mlp_reduce(
    const float* __restrict__ part, int nchunk, const double* __restrict__ lpart, double inv_n,
    float* __restrict__ grad, float* __restrict__ grad_out, double* __restrict__ loss) {
  __shared__ double sh[8][32];
  const int col = threadIdx.x & 31, row = threadIdx.x >> 5;
  const int p = blockIdx.x * 32 + col;
  double s = 0.0;
  if (p < kNPar)
#pragma unroll 4
    for (int c = row; c < nchunk; c += 8) s += (double)part[(long)c * kNPar + p];
  sh[row][col] = s;
  __syncthreads();
  if (row == 0 && p < kNPar) {
    for (int r = 1; r < 8; ++r) s += sh[r][col];
    grad[p] = (float)s;
    if (grad_out) grad_out[p] = (float)s;
  }
  if (blockIdx.x == 0 && row == 1) {  // the loss
    double v = 0.0;
    for (int c = col; c < nchunk; c += 32) v += lpart[c];
    v = warp_sum(v);
    if (col == 0) *loss = v * inv_n;
  }
}

// Adam (beta1 0.9, beta2 0.999, eps 1e-8); outputs 3..7 stay zero.
__global__ void k_adam(float* __restrict__ par, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ g, float lr, float bc1, float bc2) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= kNPar) return;
  bool frozen = false;
  if (p >= kOffW4 && p < kOffB4) frozen = ((p - kOffW4) % kNO) >= 3;
  if (p >= kOffB4) frozen = (p - kOffB4) >= 3;
  if (frozen) {
    par[p] = 0.f;
    return;
  }
  const float gi = g[p];
  const float mi = 0.9f * m[p] + 0.1f * gi;
  const float vi = 0.999f * v[p] + 0.001f * gi * gi;
  m[p] = mi;
  v[p] = vi;
  par[p] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + 1e-8f);
}

// ------------------------------------------------------------------ host

static uint64_t splitmix64(uint64_t& s) {
  uint64_t z = (s += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Launch geometry: functions of N only, so that the partial sums and hence the
// results do not depend on the device.
static long fwd_blocks(long N) { return std::min(cdiv(N, (long)kFwdWarps * kFwdRows), 152L); }
static void train_geometry(long N, long& grid, long& per) {
  const long ntile = cdiv(N, (long)kTA);
  per = cdiv(ntile, (long)kTGrid);
  grid = per > 0 ? cdiv(ntile, per) : 0;
}

// Buffer of mls6_mlp_apply (features of N atoms).
static int grow(Mlp* m, long N) {
  if (N <= m->cap) return MLS6_OK;
  if (m->d_X) cudaFree(m->d_X);
  m->d_X = nullptr;
  m->cap = 0;
  if (cudaMalloc((void**)&m->d_X, sizeof(__nv_bfloat16) * kNF * N) != cudaSuccess) {
    m->d_X = nullptr;
    return MLS6_ERR_NOMEM;
  }
  m->cap = N;
  return MLS6_OK;
}

// Buffers of the gradient (the same for every batch).
static int grow_train(Mlp* m) {
  if (!m->d_part &&
      cudaMalloc((void**)&m->d_part, sizeof(float) * kNPar * kTGrid) != cudaSuccess) {
    m->d_part = nullptr;
    return MLS6_ERR_NOMEM;
  }
  if (!m->d_lpart && cudaMalloc((void**)&m->d_lpart, sizeof(double) * kTGrid) != cudaSuccess) {
    m->d_lpart = nullptr;
    return MLS6_ERR_NOMEM;
  }
  return MLS6_OK;
}

static int repack(Mlp* m) {
  k_mlp_pack<<<cdiv(kPkAll, 256), 256, 0, m->stream>>>(m->d_par, m->d_pack);
  CK(cudaGetLastError());
  return MLS6_OK;
}

template <typename T>
static int forward(Mlp* m, const void* X, long N, float* Y, Correction<T> C, cudaStream_t st) {
  if (N <= 0) return MLS6_OK;
  k_mlp_fwd<T><<<fwd_blocks(N), 32 * kFwdWarps, sizeof(FwdShared), st>>>(
      (const __nv_bfloat16*)X, N, (reinterpret_cast<uintptr_t>(X) & 15) == 0, m->d_pack, m->d_par,
      Y, C);
  CK(cudaGetLastError());
  return MLS6_OK;
}

// Loss and gradient into d_loss, d_grad and, where grad is given, grad: by
// the reduction itself where a kernel can store there, by a copy otherwise.
static int gradient(Mlp* m, const void* X, const float* T, long N, float* grad) {
  int rc = grow_train(m);
  if (rc) return rc;
  long nch, per;
  train_geometry(N, nch, per);
  const bool direct =
      grad && (reinterpret_cast<uintptr_t>(grad) & 3) == 0 && kernel_addressable(grad);
  k_mlp_train<<<nch, 256, sizeof(TrainShared), m->stream>>>(
      (const __nv_bfloat16*)X, T, N, per, 1.0f / (float)N, m->d_pack, m->d_par, m->d_part,
      m->d_lpart);
  k_mlp_reduce<<<cdiv(kNPar, 32), 256, 0, m->stream>>>(m->d_part, (int)nch, m->d_lpart,
                                                      1.0 / (double)N, m->d_grad,
                                                      direct ? grad : nullptr, m->d_loss);
  CK(cudaGetLastError());
  if (grad && !direct)
    CK(cudaMemcpyAsync(grad, m->d_grad, sizeof(float) * kNPar, cudaMemcpyDeviceToDevice,
                       m->stream));
  return MLS6_OK;
}

static int read_loss(Mlp* m, double* loss) {
  if (!loss) return MLS6_OK;
  CK(cudaMemcpyAsync(loss, m->d_loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream));
  CK(cudaStreamSynchronize(m->stream));
  return MLS6_OK;
}

static void free_mlp(Mlp* m) {
  if (!m) return;
  void* bufs[] = {m->d_par, m->d_m, m->d_v, m->d_pack, m->d_norm, m->d_X, m->d_part, m->d_lpart,
                  m->d_grad, m->d_loss};
  for (void* b : bufs)
    if (b) cudaFree(b);
  delete m;
}

template <typename T>
static int features_t(Plan* p, Mlp* m, void* out, int f32, bool sorted_out, cudaStream_t st) {
  const Level& L1 = p->lv[1];
  const int N = (int)p->N;
  if (N == 0) return MLS6_OK;
  auto kern = f32 ? k_features<T, true> : k_features<T, false>;
  kern<<<cdiv(N, kFA), 3 * kFA, 0, st>>>(
      (const Vec4<T>*)p->d_sorted, p->d_sorted_idx, N, (const T*)level1_potential(p), L1.n[0], L1.n[1],
      L1.n[2], (T)(1.0 / L1.h[0]), (T)(1.0 / L1.h[1]), (T)(1.0 / L1.h[2]), m->d_norm, out,
      sorted_out ? 1 : 0);
  CK(cudaGetLastError());
  return MLS6_OK;
}

// Features in sorted order, then the network with the correction as its last
// step, on the plan's stream.
template <typename T> static int apply_t(Plan* p, Mlp* m, void* forces) {
  const int rc = features_t<T>(p, m, m->d_X, 0, true, p->stream);
  if (rc) return rc;
  return forward(m, m->d_X, p->N, nullptr,
                 Correction<T>{(const Vec4<T>*)p->d_sorted, p->d_sorted_idx, (T)m->out_scale,
                               (T*)forces},
                 p->stream);
}

}  // namespace mls6

using namespace mls6;

extern "C" {

int mls6_mlp_n_params(void) { return kNPar; }

int mls6_mlp_create(mls6_mlp_t** out, uint64_t seed) {
  if (!out) return MLS6_ERR_ARG;
  *out = nullptr;
  Mlp* m = new (std::nothrow) Mlp();
  if (!m) return MLS6_ERR_NOMEM;
  if (cudaMalloc((void**)&m->d_par, sizeof(float) * kNPar) != cudaSuccess ||
      cudaMalloc((void**)&m->d_m, sizeof(float) * kNPar) != cudaSuccess ||
      cudaMalloc((void**)&m->d_v, sizeof(float) * kNPar) != cudaSuccess ||
      cudaMalloc((void**)&m->d_grad, sizeof(float) * kNPar) != cudaSuccess ||
      cudaMalloc((void**)&m->d_pack, sizeof(uint2) * kPkAll) != cudaSuccess ||
      cudaMalloc((void**)&m->d_norm, sizeof(float) * 2 * kNF) != cudaSuccess ||
      cudaMalloc((void**)&m->d_loss, sizeof(double)) != cudaSuccess) {
    free_mlp(m);
    return MLS6_ERR_NOMEM;
  }
  // shared memory above 48 KB
  const auto dyn = cudaFuncAttributeMaxDynamicSharedMemorySize;
  if (cudaFuncSetAttribute(k_mlp_train, dyn, (int)sizeof(TrainShared)) != cudaSuccess ||
      cudaFuncSetAttribute(k_mlp_fwd<float>, dyn, (int)sizeof(FwdShared)) != cudaSuccess ||
      cudaFuncSetAttribute(k_mlp_fwd<double>, dyn, (int)sizeof(FwdShared)) != cudaSuccess) {
    free_mlp(m);
    return MLS6_ERR_CUDA;
  }
  // Glorot-uniform weights from SplitMix64, zero biases, outputs 3..7 zero
  std::vector<float> p(kNPar, 0.f);
  uint64_t s = seed;
  auto fill = [&](int off, int K, int Nn, int used) {
    const double lim = std::sqrt(6.0 / (K + used));
    for (int k = 0; k < K; ++k)
      for (int n = 0; n < Nn; ++n) {
        const double u = (double)(splitmix64(s) >> 11) * 0x1.0p-53;
        p[off + k * Nn + n] = n < used ? (float)((2.0 * u - 1.0) * lim) : 0.f;
      }
  };
  fill(kOffW1, kNF, kH, kH);
  fill(kOffW2, kH, kH, kH);
  fill(kOffW3, kH, kH, kH);
  fill(kOffW4, kH, kNO, 3);
  std::vector<float> norm(2 * kNF, 0.f);
  for (int j = 0; j < kNF; ++j) norm[kNF + j] = 1.f;
  if (cudaMemcpy(m->d_par, p.data(), sizeof(float) * kNPar, cudaMemcpyHostToDevice) !=
          cudaSuccess ||
      cudaMemcpy(m->d_norm, norm.data(), sizeof(float) * 2 * kNF, cudaMemcpyHostToDevice) !=
          cudaSuccess ||
      cudaMemset(m->d_m, 0, sizeof(float) * kNPar) != cudaSuccess ||
      cudaMemset(m->d_v, 0, sizeof(float) * kNPar) != cudaSuccess || repack(m) != MLS6_OK ||
      cudaStreamSynchronize(m->stream) != cudaSuccess) {
    free_mlp(m);
    return MLS6_ERR_CUDA;
  }
  *out = reinterpret_cast<mls6_mlp_t*>(m);
  return MLS6_OK;
}

int mls6_mlp_set_stream(mls6_mlp_t* mm, void* stream) {
  if (!mm) return MLS6_ERR_ARG;
  reinterpret_cast<Mlp*>(mm)->stream = (cudaStream_t)stream;
  return MLS6_OK;
}

int mls6_mlp_get_params(const mls6_mlp_t* mm, float* host, int n) {
  if (!mm || !host || n != kNPar) return MLS6_ERR_ARG;
  const Mlp* m = reinterpret_cast<const Mlp*>(mm);
  CK(cudaStreamSynchronize(m->stream));
  CK(cudaMemcpy(host, m->d_par, sizeof(float) * kNPar, cudaMemcpyDeviceToHost));
  return MLS6_OK;
}

int mls6_mlp_set_params(mls6_mlp_t* mm, const float* host, int n) {
  if (!mm || !host || n != kNPar) return MLS6_ERR_ARG;
  Mlp* m = reinterpret_cast<Mlp*>(mm);
  CK(cudaStreamSynchronize(m->stream));
  CK(cudaMemcpy(m->d_par, host, sizeof(float) * kNPar, cudaMemcpyHostToDevice));
  CK(cudaMemset(m->d_m, 0, sizeof(float) * kNPar));
  CK(cudaMemset(m->d_v, 0, sizeof(float) * kNPar));
  m->step = 0;
  return repack(m);
}

int mls6_mlp_set_norm(mls6_mlp_t* mm, const float* shift, const float* scale, float out_scale) {
  if (!mm || !shift || !scale || !std::isfinite(out_scale)) return MLS6_ERR_ARG;
  Mlp* m = reinterpret_cast<Mlp*>(mm);
  std::vector<float> norm(2 * kNF);
  for (int j = 0; j < kNF; ++j) {
    norm[j] = shift[j];
    norm[kNF + j] = scale[j];
  }
  CK(cudaStreamSynchronize(m->stream));
  CK(cudaMemcpy(m->d_norm, norm.data(), sizeof(float) * 2 * kNF, cudaMemcpyHostToDevice));
  m->out_scale = out_scale;
  return MLS6_OK;
}

int mls6_mlp_features(mls6_plan_t* plan, const mls6_mlp_t* mm, void* out, int fmt) {
  if (!plan || !mm || (fmt != 0 && fmt != 1)) return MLS6_ERR_ARG;
  Plan* p = reinterpret_cast<Plan*>(plan);
  if (p->order != 3) return MLS6_ERR_ORDER;  // features are defined on the cubic basis
  if (p->N > 0 && !kernel_addressable(out)) return MLS6_ERR_ARG;
  Mlp* m = const_cast<Mlp*>(reinterpret_cast<const Mlp*>(mm));
  return p->prec == MLS6_FP64 ? features_t<double>(p, m, out, fmt, false, p->stream)
                              : features_t<float>(p, m, out, fmt, false, p->stream);
}

int mls6_mlp_forward(mls6_mlp_t* mm, const void* X, int64_t N, float* Y) {
  if (!mm || N < 0 || (N > 0 && (!kernel_addressable(X) || !kernel_addressable(Y))))
    return MLS6_ERR_ARG;
  Mlp* m = reinterpret_cast<Mlp*>(mm);
  return forward(m, X, N, Y, Correction<float>{}, m->stream);
}

int mls6_mlp_grad(mls6_mlp_t* mm, const void* X, const float* T, int64_t N, float* grad,
                  double* loss) {
  if (!mm || N < 1 || !kernel_addressable(X) || !kernel_addressable(T) ||
      (reinterpret_cast<uintptr_t>(X) & 15))
    return MLS6_ERR_ARG;
  Mlp* m = reinterpret_cast<Mlp*>(mm);
  int rc = gradient(m, X, T, N, grad);
  if (rc) return rc;
  return read_loss(m, loss);
}

int mls6_mlp_train_step(mls6_mlp_t* mm, const void* X, const float* T, int64_t N, float lr,
                        double* loss) {
  if (!mm || N < 1 || !kernel_addressable(X) || !kernel_addressable(T) || !(lr > 0.f) ||
      (reinterpret_cast<uintptr_t>(X) & 15))
    return MLS6_ERR_ARG;
  Mlp* m = reinterpret_cast<Mlp*>(mm);
  int rc = gradient(m, X, T, N, nullptr);
  if (rc) return rc;
  m->step += 1;
  const float bc1 = 1.f - (float)std::pow(0.9, (double)m->step);
  const float bc2 = 1.f - (float)std::pow(0.999, (double)m->step);
  k_adam<<<cdiv(kNPar, 256), 256, 0, m->stream>>>(m->d_par, m->d_m, m->d_v, m->d_grad, lr, bc1,
                                                  bc2);
  CK(cudaGetLastError());
  rc = repack(m);
  if (rc) return rc;
  return read_loss(m, loss);
}

int mls6_mlp_apply(mls6_plan_t* plan, mls6_mlp_t* mm, void* forces) {
  if (!plan || !mm) return MLS6_ERR_ARG;
  Plan* p = reinterpret_cast<Plan*>(plan);
  Mlp* m = reinterpret_cast<Mlp*>(mm);
  if (p->order != 3) return MLS6_ERR_ORDER;
  const long N = p->N;
  if (N == 0) return MLS6_OK;
  if (!kernel_addressable(forces)) return MLS6_ERR_ARG;
  int rc = grow(m, N);
  if (rc) return rc;
  return p->prec == MLS6_FP64 ? apply_t<double>(p, m, forces) : apply_t<float>(p, m, forces);
}

void mls6_mlp_destroy(mls6_mlp_t* mm) { free_mlp(reinterpret_cast<Mlp*>(mm)); }

}  // extern "C"
