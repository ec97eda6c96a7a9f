// Grid part of an evaluation in Fourier space.  Between the anterpolated
// coefficients q^1 and the total potential e^{1,tot} on the finest grid every
// step of Sec. II.B is linear and periodic: restriction, the level stencils
// (Eq. evaluation), the coarsest level (Eq. last-grid-periodic-transformed)
// and prolongation.  In the discrete Fourier transform of the finest grid
// they become products with real factors that tables hold:
//   restriction    q^{k+1}(x) = 1/8 sum over the 8 aliases x + a n_{k+1} of
//                  w(x) q^k, w(x) = prod_d sum_o Phi(o/2) cos(2 pi x_d o/n_k,d)
//   evaluation     e^k(x) = K_k(x) q^k(x), K_k the transform of g_k's taps; on
//                  level k < l it is level 1's at 2^(k-1) x, times 2^(-6(k-1))
//   prolongation   e^{k,tot}(x) = e^k(x) + w(x) e^{k+1,tot}(x mod n_{k+1})
//   virial         W_ab = 1/2 sum_k 1/N_k sum_x |q^k(x)|^2 V_ab,k(x), V_ab,k
//                  the transform of the taps g_k'/r r_a r_b
// The direct kernels (mls6_grid.cu, the tensor-core stencils) compute the same
// grids node by node; they stay for grids this form does not take, for plans
// that ask for a stencil kernel, for mls6_debug_grid, and for evaluations with
// thin phases, whose potentials the transforms would round too coarsely: there
// (k_thin_body, mls6_bin.cu) every kernel here returns at once and the direct
// form runs in one launch behind them (mls6_direct.cu).
//
// Why: the direct stencils cost ~1000 taps per node (14 operations each with
// the virial) and the hierarchy 2 l launches of ever smaller grids; the
// transforms cost ~100 operations per node and five launches for all levels.
// Restriction to prolongation, direct -> here: 112^3, 5 levels, mixed 344 ->
// 89 us; 48^3 FP64 798 -> 98 us; 12^3 FP64 438 -> 37 us (eight 8^3 tiles kept
// eight SMs busy at the FP64 rate); 16 x 16 x 44 FP32 67 -> 28 us (latency of
// seven launches).  Bound now by latency: few blocks (one per plane: 112 of
// 152 SMs) of dependent shared-memory passes, 45% of the issue slots.
//
//   k_spec_fwd   a plane z: fixed-point sums -> q^1, real transform along x
//                (two reals packed as one complex), then along y
//   k_spec_z     kSpecCols columns: transform along z (forward, and inverse)
//   k_spec_tree  the frequencies that are equal modulo the coarsest grid form
//                a closed set (8^(l-1) of them): one block takes a set through
//                all levels, down and up, in shared memory
//   k_spec_inv   a plane z: inverse along y and x -> e^{1,tot}
//
// The x axis keeps frequencies 0..n0/2 (the input is real).  Transforms are
// Stockham passes of radix 2, 3, 4, 5, 7, 8, 11, 13, 17, 19 between two
// shared-memory buffers, many lines at once with the line index fastest over
// the threads (rows have an odd pitch: no bank conflicts).  All results are
// independent of the number of threads, except the virial's partial sums,
// which fix 256.
#include <algorithm>
#include <cmath>
#include <vector>

#include "mls6_device.cuh"

namespace mls6 {

template <typename T> struct alignas(2 * sizeof(T)) Cx {
  T x, y;
};

constexpr int kSpecThreads = 256;
constexpr int kSpecCols = 16;
constexpr int kSpecMaxLevels = 5;               // 8^4 + ... frequencies in shared memory
constexpr size_t kSpecSmemMax = 200 * 1024;

// Threads of a plane's block: the planes are few (one per z) and the passes
// wait on shared memory, so as many as the radices' registers allow.
template <typename T, int MAXR> constexpr int spec_plane_threads() {
  return MAXR == 8 ? (sizeof(T) == 4 ? 1024 : 512) : (sizeof(T) == 4 ? 512 : 256);
}

template <typename T> struct SpecArgs {
  int n[3], h0, M, pitch, RL;     // finest grid, n0/2 + 1, n0/2, odd pitch >= h0, n1 h0
  unsigned long long rad[3];      // radices, 5 bits each (x: of M), lowest first
  const Cx<T>* tw[3];             // exp(-2 pi i j / n_d), j < n_d
  const typename Fixed<T>::U* qfx;
  const int* flag;                // flag[kThin]: the direct kernels run instead
  double span;
  int lb;                         // Lorentz-Berthelot: channel = grid y index
  double lbc[7];
  Cx<T>* S;                       // [z][ky][kx], the input's transform
  Cx<T>* R;                       // the same of the result (other sets still read S)
  T* et;
  long np, ns;                    // nodes; elements of S (channel strides)
  int l, m[3];
  const T* w[3];                  // restriction / prolongation factor per axis, n_d entries
  const Vec4<T>* K;               // level 1, one octant: energy and six virial factors, padding
  int o[3];
  const double* Kt;               // coarsest level: the same seven, whole grid
  double* wpart;                  // one record per set of frequencies
  T inv_n;
};

template <typename T> __device__ __forceinline__ Cx<T> cmul(Cx<T> a, Cx<T> b) {
  return Cx<T>{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <typename T> __device__ __forceinline__ Cx<T> cadd(Cx<T> a, Cx<T> b) {
  return Cx<T>{a.x + b.x, a.y + b.y};
}
template <typename T> __device__ __forceinline__ Cx<T> csub(Cx<T> a, Cx<T> b) {
  return Cx<T>{a.x - b.x, a.y - b.y};
}
// i / d for 0 <= i < 2^20 (inv = 1.0f / d)
__device__ __forceinline__ int idiv(int i, float inv) { return (int)(((float)i + 0.5f) * inv); }

// 4-point transform in place, sg = 1 forward, -1 inverse.
template <typename T> __device__ __forceinline__ void dft4(Cx<T>& a, Cx<T>& b, Cx<T>& c, Cx<T>& d, T sg) {
  const Cx<T> s = cadd(a, c), t = csub(a, c), u = cadd(b, d), v = csub(b, d);
  a = cadd(s, u);
  c = csub(s, u);
  b = Cx<T>{t.x + sg * v.y, t.y - sg * v.x};
  d = Cx<T>{t.x - sg * v.y, t.y + sg * v.x};
}

// One Stockham pass of radix R over `lines` lines of n points (line stride
// ls, element stride es): sub-transforms of length s become ones of length
// s R.  tw: exp(-2 pi i j / (n tws)), so that tws j steps by 1/n.
template <typename T, int R>
__device__ __forceinline__ void spec_pass(const Cx<T>* a, Cx<T>* b, int lines,
                                          int ls, int n, int es, int s, const Cx<T>* tw, int tws,
                                          T sg) {
  const int nb = n / R, total = lines * nb, step = tws * (nb / s), unit = tws * nb;
  const float il = 1.0f / (float)lines, is = 1.0f / (float)s;
  for (int i = threadIdx.x; i < total; i += blockDim.x) {
    const int j = idiv(i, il), line = i - j * lines;
    const int q = idiv(j, is), k = j - q * s;
    const Cx<T>* src = a + line * ls + j * es;
    Cx<T>* dst = b + line * ls + (q * s * R + k) * es;
    Cx<T> v[R];
#pragma unroll
    for (int t = 0; t < R; ++t) v[t] = src[t * nb * es];
    if (k > 0) {
#pragma unroll
      for (int t = 1; t < R; ++t) {
        Cx<T> w = tw[t * k * step];
        w.y *= sg;
        v[t] = cmul(v[t], w);
      }
    }
    if constexpr (R == 2) {
      dst[0] = cadd(v[0], v[1]);
      dst[s * es] = csub(v[0], v[1]);
    } else if constexpr (R == 4) {
      dft4(v[0], v[1], v[2], v[3], sg);
#pragma unroll
      for (int t = 0; t < 4; ++t) dst[t * s * es] = v[t];
    } else if constexpr (R == 8) {
      dft4(v[0], v[2], v[4], v[6], sg);
      dft4(v[1], v[3], v[5], v[7], sg);
      const T h = T(0.70710678118654752440);
      const Cx<T> a1{h * (v[3].x + sg * v[3].y), h * (v[3].y - sg * v[3].x)};
      const Cx<T> a2{sg * v[5].y, -sg * v[5].x};
      const Cx<T> a3{h * (sg * v[7].y - v[7].x), -h * (v[7].y + sg * v[7].x)};
      dst[0] = cadd(v[0], v[1]);
      dst[4 * s * es] = csub(v[0], v[1]);
      dst[s * es] = cadd(v[2], a1);
      dst[5 * s * es] = csub(v[2], a1);
      dst[2 * s * es] = cadd(v[4], a2);
      dst[6 * s * es] = csub(v[4], a2);
      dst[3 * s * es] = cadd(v[6], a3);
      dst[7 * s * es] = csub(v[6], a3);
    } else {  // odd prime: X_k, X_{R-k} = v_0 + sum_j (v_j + v_{R-j}) cos -/+ i (v_j - v_{R-j}) sin
      constexpr int H = (R - 1) / 2;
      T c[H + 1], sn[H + 1];
#pragma unroll
      for (int t = 1; t <= H; ++t) {
        const Cx<T> w = tw[t * unit];
        c[t] = w.x;
        sn[t] = -sg * w.y;
      }
      Cx<T> sum = v[0];
#pragma unroll
      for (int t = 1; t <= H; ++t) {
        const Cx<T> p = v[t], m = v[R - t];
        v[t] = cadd(p, m);
        v[R - t] = csub(p, m);
        sum = cadd(sum, v[t]);
      }
      dst[0] = sum;
#pragma unroll
      for (int k2 = 1; k2 <= H; ++k2) {
        Cx<T> A = v[0], B{T(0), T(0)};
#pragma unroll
        for (int t = 1; t <= H; ++t) {
          const int m = (t * k2) % R, mm = m > H ? R - m : m;
          const T sv = m > H ? -sn[mm] : sn[mm];
          A.x += c[mm] * v[t].x;
          A.y += c[mm] * v[t].y;
          B.x += sv * v[R - t].x;
          B.y += sv * v[R - t].y;
        }
        dst[k2 * s * es] = Cx<T>{A.x + B.y, A.y - B.x};
        dst[(R - k2) * s * es] = Cx<T>{A.x - B.y, A.y + B.x};
      }
    }
  }
}

// Transform of `lines` lines from buffer a (scratch b); returns the buffer
// that holds the result.  Starts and ends with a block barrier.
template <typename T, int MAXR>
__device__ __noinline__ Cx<T>* spec_lines(Cx<T>* a, Cx<T>* b, int lines, int ls, int n, int es,
                                          unsigned long long rad, const Cx<T>* tw, int tws, T sg) {
  int s = 1;
  __syncthreads();
  for (; rad; rad >>= 5) {
    const int r = (int)(rad & 31);
    switch (r) {
      case 2: spec_pass<T, 2>(a, b, lines, ls, n, es, s, tw, tws, sg); break;
      case 3: spec_pass<T, 3>(a, b, lines, ls, n, es, s, tw, tws, sg); break;
      case 4: spec_pass<T, 4>(a, b, lines, ls, n, es, s, tw, tws, sg); break;
      case 5: spec_pass<T, 5>(a, b, lines, ls, n, es, s, tw, tws, sg); break;
      case 7: spec_pass<T, 7>(a, b, lines, ls, n, es, s, tw, tws, sg); break;
      case 8: spec_pass<T, 8>(a, b, lines, ls, n, es, s, tw, tws, sg); break;
      default:
        if constexpr (MAXR > 8) switch (r) {
          case 11: spec_pass<T, 11>(a, b, lines, ls, n, es, s, tw, tws, sg); break;
          case 13: spec_pass<T, 13>(a, b, lines, ls, n, es, s, tw, tws, sg); break;
          case 17: spec_pass<T, 17>(a, b, lines, ls, n, es, s, tw, tws, sg); break;
          default: spec_pass<T, 19>(a, b, lines, ls, n, es, s, tw, tws, sg); break;
        }
    }
    __syncthreads();
    Cx<T>* t = a;
    a = b;
    b = t;
    s *= r;
  }
  return a;
}

// Shared memory: two planes of n1 rows, the x and y tables.
template <typename T> __host__ __device__ inline size_t spec_plane_smem(int n0, int n1, int pitch) {
  return sizeof(Cx<T>) * (2 * (size_t)n1 * pitch + n0 + n1);
}
template <typename T> __host__ __device__ inline size_t spec_z_smem(int n2) {
  return sizeof(Cx<T>) * (2 * (size_t)n2 * kSpecCols + n2);
}
// all levels' frequencies of one set
template <typename T> __host__ __device__ inline size_t spec_tree_smem(int l) {
  size_t e = 0;
  for (int k = 0; k < l; ++k) e += (size_t)1 << (3 * k);
  return sizeof(Cx<T>) * e;
}

// The evaluation has thin phases: the direct kernels run instead.  Each body
// reads the word beside its first data and looks at it behind them, so that the
// read's latency is not added (over the five kernels 1 us at 1,000 to 3,000 atoms).
template <typename T> __device__ __forceinline__ int spec_off(const SpecArgs<T>& A) {
  return *(volatile const int*)(A.flag + kThin);
}

template <typename T, int MAXR>
__device__ __forceinline__ void spec_fwd_body(const Blk bk, int ch, const SpecArgs<T>& A,
                                              unsigned char* smem) {
  __shared__ int sexp;
  const int off = spec_off(A);
  Cx<T>* a = reinterpret_cast<Cx<T>*>(smem);
  Cx<T>* b = a + (size_t)A.n[1] * A.pitch;
  Cx<T>* wx = b + (size_t)A.n[1] * A.pitch;
  Cx<T>* wy = wx + A.n[0];
  if (threadIdx.x == 0)
    sexp = fixed_exponent<T>(A.flag, A.span, A.lb ? ch : -1, A.lb ? A.lbc[ch] : 0.0);
  for (int i = threadIdx.x; i < A.n[0]; i += blockDim.x) wx[i] = A.tw[0][i];
  for (int i = threadIdx.x; i < A.n[1]; i += blockDim.x) wy[i] = A.tw[1][i];
  __syncthreads();
  if (off) return;
  const T isc = Fixed<T>::pow2(-sexp);
  using U = typename Fixed<T>::U;
  using I = typename Fixed<T>::I;
  const U* q = A.qfx + (size_t)ch * A.np + (size_t)bk.x * A.n[0] * A.n[1];
  const int M = A.M, h0 = A.h0, n1 = A.n[1];
  const float iM = 1.0f / (float)M, ih = 1.0f / (float)h0;
  for (int i = threadIdx.x; i < n1 * M; i += blockDim.x) {
    const int r = idiv(i, iM), j = i - r * M;
    a[r * A.pitch + j] = Cx<T>{Fixed<T>::from_fixed((I)q[2 * i], isc),
                               Fixed<T>::from_fixed((I)q[2 * i + 1], isc)};
  }
  Cx<T>* z = spec_lines<T, MAXR>(a, b, n1, A.pitch, M, 1, A.rad[0], wx, 2, T(1));
  Cx<T>* x = z == a ? b : a;
  // packed halves -> X_k = (Z_k + Z*_{M-k})/2 - i/2 w^k (Z_k - Z*_{M-k}), k = 0 .. M
  for (int i = threadIdx.x; i < n1 * h0; i += blockDim.x) {
    const int r = idiv(i, ih), k = i - r * h0;
    const Cx<T> p = z[r * A.pitch + (k == M ? 0 : k)], m = z[r * A.pitch + (k == 0 ? 0 : M - k)];
    const Cx<T> e{T(0.5) * (p.x + m.x), T(0.5) * (p.y - m.y)};
    const Cx<T> d{T(0.5) * (p.x - m.x), T(0.5) * (p.y + m.y)};
    const Cx<T> o = cmul(wx[k], Cx<T>{d.y, -d.x});
    x[r * A.pitch + k] = cadd(e, o);
  }
  Cx<T>* y = spec_lines<T, MAXR>(x, z, h0, 1, n1, A.pitch, A.rad[1], wy, 1, T(1));
  Cx<T>* S = A.S + (size_t)ch * A.ns + (size_t)bk.x * A.RL;
  for (int i = threadIdx.x; i < n1 * h0; i += blockDim.x) {
    const int r = idiv(i, ih), k = i - r * h0;
    S[i] = y[r * A.pitch + k];
  }
}

template <typename T, int MAXR>
__device__ __forceinline__ void spec_z_body(const Blk bk, int ch, const SpecArgs<T>& A, T sg,
                                            unsigned char* smem) {
  Cx<T>* a = reinterpret_cast<Cx<T>*>(smem);
  Cx<T>* b = a + (size_t)A.n[2] * kSpecCols;
  Cx<T>* wz = b + (size_t)A.n[2] * kSpecCols;
  const int off = spec_off(A);
  const int n2 = A.n[2], c0 = bk.x * kSpecCols, nc = min(kSpecCols, A.RL - c0);
  Cx<T>* S = (sg > T(0) ? A.S : A.R) + (size_t)ch * A.ns + c0;
  for (int i = threadIdx.x; i < n2; i += blockDim.x) wz[i] = A.tw[2][i];
  for (int i = threadIdx.x; i < n2 * kSpecCols; i += blockDim.x) {
    const int z = i / kSpecCols, c = i % kSpecCols;
    a[i] = c < nc ? S[(size_t)z * A.RL + c] : Cx<T>{T(0), T(0)};
  }
  if (off) return;
  const Cx<T>* r = spec_lines<T, MAXR>(a, b, kSpecCols, 1, n2, kSpecCols, A.rad[2], wz, 1, sg);
  for (int i = threadIdx.x; i < n2 * kSpecCols; i += blockDim.x) {
    const int z = i / kSpecCols, c = i % kSpecCols;
    if (c < nc) S[(size_t)z * A.RL + c] = r[i];
  }
}

template <typename T, int MAXR>
__device__ __forceinline__ void spec_inv_body(const Blk bk, int ch, const SpecArgs<T>& A,
                                              unsigned char* smem) {
  Cx<T>* a = reinterpret_cast<Cx<T>*>(smem);
  Cx<T>* b = a + (size_t)A.n[1] * A.pitch;
  Cx<T>* wx = b + (size_t)A.n[1] * A.pitch;
  Cx<T>* wy = wx + A.n[0];
  const int off = spec_off(A);
  for (int i = threadIdx.x; i < A.n[0]; i += blockDim.x) wx[i] = A.tw[0][i];
  for (int i = threadIdx.x; i < A.n[1]; i += blockDim.x) wy[i] = A.tw[1][i];
  const int M = A.M, h0 = A.h0, n1 = A.n[1];
  const float iM = 1.0f / (float)M, ih = 1.0f / (float)h0;
  const Cx<T>* S = A.R + (size_t)ch * A.ns + (size_t)bk.x * A.RL;
  for (int i = threadIdx.x; i < n1 * h0; i += blockDim.x) {
    const int r = idiv(i, ih), k = i - r * h0;
    a[r * A.pitch + k] = S[i];
  }
  if (off) return;
  Cx<T>* x = spec_lines<T, MAXR>(a, b, h0, 1, n1, A.pitch, A.rad[1], wy, 1, T(-1));
  Cx<T>* z = x == a ? b : a;
  // Z_k = (X_k + X*_{M-k}) + i w^-k (X_k - X*_{M-k}), k = 0 .. M-1
  for (int i = threadIdx.x; i < n1 * M; i += blockDim.x) {
    const int r = idiv(i, iM), k = i - r * M;
    const Cx<T> p = x[r * A.pitch + k], m = x[r * A.pitch + M - k];
    const Cx<T> e{p.x + m.x, p.y - m.y}, d{p.x - m.x, p.y + m.y};
    const Cx<T> w{wx[k].x, -wx[k].y}, o = cmul(w, d);
    z[r * A.pitch + k] = Cx<T>{e.x - o.y, e.y + o.x};
  }
  const Cx<T>* v = spec_lines<T, MAXR>(z, x, n1, A.pitch, M, 1, A.rad[0], wx, 2, T(-1));
  Cx<T>* et = reinterpret_cast<Cx<T>*>(A.et + (size_t)ch * A.np + (size_t)bk.x * A.n[0] * n1);
  for (int i = threadIdx.x; i < n1 * M; i += blockDim.x) {
    const int r = idiv(i, iM), j = i - r * M;
    et[i] = v[r * A.pitch + j];
  }
}

template <typename T, bool VIR>
__device__ __forceinline__ void spec_tree_body(const Blk bk, int ch, const SpecArgs<T>& A,
                                               unsigned char* smem) {
  __shared__ double red[32 * 6];
  Cx<T>* q = reinterpret_cast<Cx<T>*>(smem);
  const int l = A.l, lg = l - 1, n0 = A.n[0], n1 = A.n[1], n2 = A.n[2];
  const int c0 = bk.x % A.m[0], c1 = bk.x / A.m[0] % A.m[1], c2 = bk.x / (A.m[0] * A.m[1]);
  const int skip = spec_off(A);
  const Cx<T>* S = A.S + (size_t)ch * A.ns;
  Cx<T>* out = A.R + (size_t)ch * A.ns;
  const int E1 = 1 << (3 * lg);
  for (int e = threadIdx.x; e < E1; e += blockDim.x) {
    const int k0 = c0 + A.m[0] * (e & ((1 << lg) - 1));
    const int k1 = c1 + A.m[1] * (e >> lg & ((1 << lg) - 1)), k2 = c2 + A.m[2] * (e >> (2 * lg));
    if (k0 < A.h0) {
      q[e] = S[(size_t)k2 * A.RL + k1 * A.h0 + k0];
    } else {  // the conjugate's place
      const int j1 = k1 ? n1 - k1 : 0, j2 = k2 ? n2 - k2 : 0;
      const Cx<T> v = S[(size_t)j2 * A.RL + j1 * A.h0 + (n0 - k0)];
      q[e] = Cx<T>{v.x, -v.y};
    }
  }
  if (skip) return;
  __syncthreads();
  // down: q^{k+1} from the aliases of q^k
  int off = 0;
  for (int k = 1; k < l; ++k) {
    const int b = l - k, h = b - 1, o1 = off + (1 << (3 * b));  // side 2^b -> 2^h
    for (int e = threadIdx.x; e < 1 << (3 * h); e += blockDim.x) {
      const int t0 = e & ((1 << h) - 1), t1 = e >> h & ((1 << h) - 1), t2 = e >> (2 * h);
      T w0[2], w1[2], w2[2];
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        w0[a] = T(0.5) * A.w[0][(c0 + A.m[0] * (t0 + (a << h))) << (k - 1)];
        w1[a] = T(0.5) * A.w[1][(c1 + A.m[1] * (t1 + (a << h))) << (k - 1)];
        w2[a] = T(0.5) * A.w[2][(c2 + A.m[2] * (t2 + (a << h))) << (k - 1)];
      }
      Cx<T> s{T(0), T(0)};
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        const int x = a & 1, y = a >> 1 & 1, z = a >> 2;
        const Cx<T> v =
            q[off + (t0 + (x << h)) + ((t1 + (y << h)) << b) + ((t2 + (z << h)) << (2 * b))];
        const T w = w0[x] * w1[y] * w2[z];
        s.x += w * v.x;
        s.y += w * v.y;
      }
      q[o1 + e] = s;
    }
    __syncthreads();
    off = o1;
  }
  // coarsest level in FP64, its virial added to the record behind the levels' sum
  double wt[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};  // (thread 0)
  T wv[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
  const int npt = A.m[0] * A.m[1] * A.m[2];
  if (threadIdx.x == 0) {
    const Cx<T> v = q[off];
    if (VIR) {
      const double p = 0.5 / npt * ((double)v.x * v.x + (double)v.y * v.y);
#pragma unroll
      for (int c = 0; c < 6; ++c) wt[c] = p * A.Kt[(size_t)(c + 1) * npt + bk.x];
    }
    const double t = A.Kt[bk.x];
    q[off] = Cx<T>{(T)(t * v.x), (T)(t * v.y)};
  }
  __syncthreads();
  // up: e^{k,tot} in place of q^k
  for (int k = l - 1; k >= 1; --k) {
    const int b = l - k, h = b - 1, o1 = off;
    off -= 1 << (3 * b);
    T sc = T(1);
    for (int j = 1; j < k; ++j) sc *= T(1.0 / 64.0);
    const T hs = T(0.5) * sc / (T)((long)npt << (3 * b));
    for (int e = threadIdx.x; e < 1 << (3 * b); e += blockDim.x) {
      const int t0 = e & ((1 << b) - 1), t1 = e >> b & ((1 << b) - 1), t2 = e >> (2 * b);
      const int k0 = c0 + A.m[0] * t0, k1 = c1 + A.m[1] * t1, k2 = c2 + A.m[2] * t2;
      const int i0 = k0 << (k - 1), i1 = k1 << (k - 1), i2 = k2 << (k - 1);
      const int j0 = min(i0, n0 - i0), j1 = min(i1, n1 - i1), j2 = min(i2, n2 - i2);
      const Vec4<T>* K = A.K + 2 * (j0 + (size_t)A.o[0] * (j1 + (size_t)A.o[1] * j2));
      const Vec4<T> Ka = K[0];
      const Cx<T> v = q[off + e];
      if (VIR) {
        const T p = (hs * v.x) * v.x + (hs * v.y) * v.y;  // |v|^2 ~ (N c)^2 alone may overflow
        const Vec4<T> Kb = K[1];
        wv[0] += p * Ka.y;
        wv[1] += p * Ka.z;
        wv[2] += p * Ka.w;
        const bool f0 = i0 != j0, f1 = i1 != j1, f2 = i2 != j2;  // odd factors of a mirrored axis
        wv[3] += (f0 != f1 ? -p : p) * Kb.x;
        wv[4] += (f0 != f2 ? -p : p) * Kb.y;
        wv[5] += (f1 != f2 ? -p : p) * Kb.z;
      }
      const T g = sc * Ka.x, w = A.w[0][i0] * A.w[1][i1] * A.w[2][i2];
      const int hm = (1 << h) - 1;
      const Cx<T> u = q[o1 + (t0 & hm) + ((t1 & hm) << h) + ((t2 & hm) << (2 * h))];
      const Cx<T> r{g * v.x + w * u.x, g * v.y + w * u.y};
      if (k > 1)
        q[off + e] = r;
      else if (k0 < A.h0)
        out[(size_t)k2 * A.RL + k1 * A.h0 + k0] = Cx<T>{A.inv_n * r.x, A.inv_n * r.y};
    }
    __syncthreads();
  }
  if (VIR) {
    double ws[6];
    block_sum_lo<T, 6>(wv, ws, red);
    if (threadIdx.x == 0)
      for (int c = 0; c < 6; ++c) A.wpart[6 * (size_t)bk.x + c] = ws[c] + wt[c];
  }
}

#ifndef MLS6_DEVICE_ONLY
template <typename T, int MAXR>
__global__ void __launch_bounds__(spec_plane_threads<T, MAXR>()) k_spec_fwd(SpecArgs<T> A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_begin();
  spec_fwd_body<T, MAXR>(Blk::self(), blockIdx.y, A, smem_raw);
}
template <typename T, int MAXR>
__global__ void __launch_bounds__(kSpecThreads, MAXR == 8 && sizeof(T) == 4 ? 4 : 1)
    k_spec_z(SpecArgs<T> A, T sg) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_begin();
  spec_z_body<T, MAXR>(Blk::self(), blockIdx.y, A, sg, smem_raw);
}
template <typename T, bool VIR>
__global__ void __launch_bounds__(kSpecThreads) k_spec_tree(SpecArgs<T> A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_begin();
  spec_tree_body<T, VIR>(Blk::self(), blockIdx.y, A, smem_raw);
}
template <typename T, int MAXR>
__global__ void __launch_bounds__(spec_plane_threads<T, MAXR>()) k_spec_inv(SpecArgs<T> A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_begin();
  spec_inv_body<T, MAXR>(Blk::self(), blockIdx.y, A, smem_raw);
}
#endif  // MLS6_DEVICE_ONLY

// ------------------------------------------------------------------ host

// Kernel arguments of a plan (one channel, or the seven of Lorentz-Berthelot).
template <typename T> static SpecArgs<T> spec_args(const Plan* p, bool lb) {
  SpecArgs<T> A;
  const Level& L1 = p->lv[1];
  for (int d = 0; d < 3; ++d) {
    A.n[d] = L1.n[d];
    A.m[d] = p->lv[p->levels].n[d];
    A.o[d] = L1.n[d] / 2 + 1;
    A.rad[d] = p->spec_rad[d];
  }
  A.M = A.n[0] / 2;
  A.h0 = A.M + 1;
  A.pitch = A.h0 | 1;
  A.RL = A.n[1] * A.h0;
  A.np = L1.np;
  A.ns = (long)A.RL * A.n[2];
  A.l = p->levels;
  const Cx<T>* tw = reinterpret_cast<const Cx<T>*>(p->d_spec_tw);
  A.K = reinterpret_cast<const Vec4<T>*>(p->d_spec_tab);
  const T* w = reinterpret_cast<const T*>(A.K + 2 * (size_t)A.o[0] * A.o[1] * A.o[2]);
  for (int d = 0; d < 3; ++d) {
    A.tw[d] = tw;
    A.w[d] = w;
    tw += A.n[d];
    w += A.n[d];
  }
  A.Kt = p->d_spec_top;
  A.flag = p->d_flag;
  A.span = support_span(p);
  A.lb = lb ? 1 : 0;
  for (int c = 0; c < 7; ++c) A.lbc[c] = lb_coef(c);
  A.qfx = reinterpret_cast<const typename Fixed<T>::U*>(lb ? p->d_lbq : p->d_q1fx);
  A.S = reinterpret_cast<Cx<T>*>(lb ? p->d_lbs : p->d_spec_s);
  A.R = A.S + (lb ? 7 : 1) * A.ns;
  A.et = reinterpret_cast<T*>(lb ? p->d_lbpot : p->d_et[1]);
  A.wpart = p->d_wpart + 6 * p->wpart_spec;
  A.inv_n = (T)(1.0 / (double)L1.np);
  return A;
}

#ifndef MLS6_DEVICE_ONLY  // host code, left out where another unit includes this file

// Radices of n, 5 bits each; 0 radices for n = 1; false if a prime above 19 divides n.
static bool spec_radices(int n, unsigned long long* out) {
  *out = 0;
  int at = 0;
  auto put = [&](int r) {
    *out |= (unsigned long long)r << (5 * at++);
    n /= r;
  };
  int e = 0;
  while (n >> e > 1 && (n >> e) % 2 == 0) ++e;
  while (e > 0) {  // 16 as 4 x 4 rather than 8 x 2
    const int b = e == 1 ? 1 : (e == 2 || e == 4) ? 2 : 3;
    put(1 << b);
    e -= b;
  }
  for (int r : {3, 5, 7, 11, 13, 17, 19})
    while (n % r == 0) put(r);
  return n == 1 && at <= 12;
}

// The spectral form takes hierarchies of 2 to 5 levels whose axes have prime
// factors up to 19 and whose planes fit in shared memory, unless a mixed plan
// asks for a stencil kernel.
bool spectral_eligible(const Plan* p) {
  if (p->N <= 0 || p->levels < 2 || p->levels > kSpecMaxLevels) return false;
  // a mixed plan's request: the CUDA-core stencil, or the tensor cores where they apply
  if (p->prec == MLS6_MIXED &&
      (p->stencil_req == 1 || (p->stencil_req == 2 && (p->stencil_mma || p->stencil_tc))))
    return false;
  const int* n = p->lv[1].n;
  unsigned long long r;
  if (n[0] % 2 || !spec_radices(n[0] / 2, &r) || !spec_radices(n[1], &r) || !spec_radices(n[2], &r))
    return false;
  const int pitch = (n[0] / 2 + 1) | 1;
  const bool d = p->prec == MLS6_FP64;
  const size_t pl = d ? spec_plane_smem<double>(n[0], n[1], pitch)
                      : spec_plane_smem<float>(n[0], n[1], pitch);
  const size_t z = d ? spec_z_smem<double>(n[2]) : spec_z_smem<float>(n[2]);
  return pl <= kSpecSmemMax && z <= kSpecSmemMax;
}

// Real transform of taps that are even (or odd, from sine sums) along each
// axis, as a separable sum of cosines (sines).  Level 1: rows of constant
// (dy, dz) with dx contiguous (Plan::h_rows, h_wv).  Seven factors per
// frequency of one octant: g_1, then g_1'/r r_a r_b for xx yy zz xy xz yz (an
// off-diagonal tap is odd along two axes: -sin sin).
// Records of 8 (one or two 32-byte sectors) per frequency, x fastest.
template <typename T> static void spec_level_tables(const Plan* p, T* tab) {
  const int* n = p->lv[1].n;
  const double* h = p->lv[1].h;
  const int o0 = n[0] / 2 + 1, o1 = n[1] / 2 + 1, o2 = n[2] / 2 + 1;
  std::vector<double> cs[3], sn[3];
  for (int d = 0; d < 3; ++d) {
    cs[d].resize(n[d]);
    sn[d].resize(n[d]);
    for (int j = 0; j < n[d]; ++j) {
      cs[d][j] = std::cos(2.0 * M_PI * j / n[d]);
      sn[d][j] = std::sin(2.0 * M_PI * j / n[d]);
    }
  }
  auto at = [&](int d, int k, int m) { return (int)(((long)k * m) % n[d]); };
  // rows with dy, dz >= 0, grouped by dz
  const int P = p->P;
  std::vector<std::vector<int>> by_z(P + 1);
  for (int r = 0; r < p->nrows; ++r)
    if (p->h_rows[4 * r] >= 0 && p->h_rows[4 * r + 1] >= 0)
      by_z[p->h_rows[4 * r + 1]].push_back(r);
  // per dz the sums over dx and dy: seven planes each
  const size_t pl = (size_t)o0 * o1;
  std::vector<int> zs;
  for (int dz = 0; dz <= P; ++dz)
    if (!by_z[dz].empty()) zs.push_back(dz);
  std::vector<double> A(4 * (size_t)o0), Pz(7 * pl * zs.size(), 0.0);
  for (size_t iz = 0; iz < zs.size(); ++iz)
    for (int r : by_z[zs[iz]]) {
      const int dy = p->h_rows[4 * r], R = p->h_rows[4 * r + 2];
      const double* wv = &p->h_wv[4 * (size_t)p->h_rows[4 * r + 3]];
      std::fill(A.begin(), A.end(), 0.0);
      for (int k = 0; k < o0; ++k)
        for (int dx = 0; dx <= R; ++dx) {
          const double* w = wv + 4 * (size_t)(dx + R);  // g, G, G dx, G dx^2
          const int i = at(0, k, dx);
          const double c = (dx ? 2.0 : 1.0) * cs[0][i];
          A[k] += w[0] * c;
          A[o0 + k] += w[1] * c;
          A[2 * o0 + k] += w[3] * c;
          A[3 * o0 + k] += w[2] * 2.0 * sn[0][i];
        }
      for (int k1 = 0; k1 < o1; ++k1) {
        const int i = at(1, k1, dy);
        const double c = (dy ? 2.0 : 1.0) * cs[1][i], s = dy * 2.0 * sn[1][i];
        double* q = &Pz[7 * pl * iz + (size_t)k1 * o0];
        for (int k = 0; k < o0; ++k) {
          const double g = A[k], G = A[o0 + k], G2 = A[2 * o0 + k], G1 = A[3 * o0 + k];
          q[k] += g * c;
          q[pl + k] += G2 * c;
          q[2 * pl + k] += G * dy * dy * c;
          q[3 * pl + k] += G * c;
          q[4 * pl + k] += G1 * s;  // odd along x and y
          q[5 * pl + k] += G1 * c;  // odd along x (and z)
          q[6 * pl + k] += G * s;   // odd along y (and z)
        }
      }
    }
  // sums over dz, one row of frequencies at a time
  std::vector<double> row((size_t)7 * o0);
  for (int k2 = 0; k2 < o2; ++k2)
    for (int k1 = 0; k1 < o1; ++k1) {
      std::fill(row.begin(), row.end(), 0.0);
      for (size_t iz = 0; iz < zs.size(); ++iz) {
        const int dz = zs[iz], i = at(2, k2, dz);
        const double c = (dz ? 2.0 : 1.0) * cs[2][i], s = dz * 2.0 * sn[2][i];
        const double f[7] = {c, c * h[0] * h[0], c * h[1] * h[1], c * dz * dz * h[2] * h[2],
                             -c * h[0] * h[1], -s * h[0] * h[2], -s * h[1] * h[2]};
        for (int ch = 0; ch < 7; ++ch) {
          const double* a = &Pz[pl * (7 * iz + ch) + (size_t)k1 * o0];
          double* q = &row[(size_t)ch * o0];
          for (int k = 0; k < o0; ++k) q[k] += f[ch] * a[k];
        }
      }
      T* out = tab + 8 * ((size_t)k2 * pl + (size_t)k1 * o0);
      for (int k = 0; k < o0; ++k)
        for (int ch = 0; ch < 7; ++ch) out[8 * (size_t)k + ch] = (T)row[(size_t)ch * o0 + k];
    }
}

// The same for the coarsest level's periodic tables (whole grid).
static void spec_top_tables(const Plan* p, std::vector<double>& Kt) {
  const Level& L = p->lv[p->levels];
  const int* n = L.n;
  Kt.assign(7 * (size_t)L.np, 0.0);
  std::vector<double> a((size_t)L.np), b((size_t)L.np);
  // axis by axis: cosine sums of an even axis, sine sums of an odd one
  static const bool odd[7][3] = {{false, false, false}, {false, false, false}, {false, false, false},
                                 {false, false, false}, {true, true, false},   {true, false, true},
                                 {false, true, true}};
  std::vector<double> wave[2][3];  // cosines, sines of 2 pi j / n
  for (int d = 0; d < 3; ++d)
    for (int j = 0; j < n[d]; ++j) {
      wave[0][d].push_back(std::cos(2.0 * M_PI * j / n[d]));
      wave[1][d].push_back(std::sin(2.0 * M_PI * j / n[d]));
    }
  for (int ch = 0; ch < 7; ++ch) {
    for (long i = 0; i < L.np; ++i)
      a[i] = ch ? p->h_top_V[(size_t)(ch - 1) * L.np + i] : p->h_top_T[i];
    long st = 1;
    for (int d = 0; d < 3; ++d) {
      for (long i = 0; i < L.np; ++i) {
        const int k = (int)(i / st % n[d]);
        const long base = i - k * st;
        const std::vector<double>& w = wave[odd[ch][d]][d];
        double s = 0.0;
        for (int m = 0; m < n[d]; ++m) s += a[base + m * st] * w[(long)k * m % n[d]];
        b[i] = s;
      }
      a.swap(b);
      st *= n[d];
    }
    for (long i = 0; i < L.np; ++i) Kt[(size_t)ch * L.np + i] = ch >= 4 ? -a[i] : a[i];
  }
}

// Shared-memory limits: properties of the kernels, shared by every plan, so
// the ceiling and not one plan's size.
template <typename T, int MAXR> static int spec_attrs() {
  const auto at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const int sm = (int)kSpecSmemMax;
  return cudaFuncSetAttribute(k_spec_fwd<T, MAXR>, at, sm) != cudaSuccess ||
         cudaFuncSetAttribute(k_spec_z<T, MAXR>, at, sm) != cudaSuccess ||
         cudaFuncSetAttribute(k_spec_tree<T, true>, at, sm) != cudaSuccess ||
         cudaFuncSetAttribute(k_spec_tree<T, false>, at, sm) != cudaSuccess ||
         cudaFuncSetAttribute(k_spec_inv<T, MAXR>, at, sm) != cudaSuccess;
}

template <typename T> int prepare_spectral(Plan* p) {
  const int* n = p->lv[1].n;
  for (int d = 0; d < 3; ++d) spec_radices(d ? n[d] : n[0] / 2, &p->spec_rad[d]);
  const size_t ntw = (size_t)n[0] + n[1] + n[2];
  std::vector<Cx<T>> tw;
  std::vector<T> tab;
  tw.reserve(ntw);
  for (int d = 0; d < 3; ++d)
    for (int j = 0; j < n[d]; ++j)
      tw.push_back(Cx<T>{(T)std::cos(2.0 * M_PI * j / n[d]), (T)-std::sin(2.0 * M_PI * j / n[d])});
  std::vector<double> Kt;
  spec_top_tables(p, Kt);
  const size_t noct = (size_t)(n[0] / 2 + 1) * (n[1] / 2 + 1) * (n[2] / 2 + 1);
  tab.reserve(8 * noct + ntw);
  tab.resize(8 * noct, T(0));
  spec_level_tables<T>(p, tab.data());
  // Phi at half-integer offsets 1/2, 3/2 (5/2)
  static const double w3[3] = {0.5625, -0.0625, 0.0};
  static const double w5[3] = {150.0 / 256.0, -25.0 / 256.0, 3.0 / 256.0};
  const double* hw = p->order == 5 ? w5 : w3;
  for (int d = 0; d < 3; ++d)
    for (int j = 0; j < n[d]; ++j) {
      double v = 1.0;
      for (int o = 0; o < 3; ++o)
        v += 2.0 * hw[o] * std::cos(2.0 * M_PI * ((long)j * (2 * o + 1) % n[d]) / n[d]);
      tab.push_back((T)v);
    }
  const long ns = (long)n[1] * (n[0] / 2 + 1) * n[2];
  if (cudaMalloc(&p->d_spec_tw, sizeof(Cx<T>) * tw.size()) != cudaSuccess ||
      cudaMalloc(&p->d_spec_tab, sizeof(T) * tab.size()) != cudaSuccess ||
      cudaMalloc((void**)&p->d_spec_top, sizeof(double) * Kt.size()) != cudaSuccess ||
      cudaMalloc(&p->d_spec_s, sizeof(Cx<T>) * 2 * ns) != cudaSuccess)
    return MLS6_ERR_NOMEM;
  const auto H2D = cudaMemcpyHostToDevice;
  if (cudaMemcpy(p->d_spec_tw, tw.data(), sizeof(Cx<T>) * tw.size(), H2D) != cudaSuccess ||
      cudaMemcpy(p->d_spec_tab, tab.data(), sizeof(T) * tab.size(), H2D) != cudaSuccess ||
      cudaMemcpy(p->d_spec_top, Kt.data(), sizeof(double) * Kt.size(), H2D) != cudaSuccess)
    return MLS6_ERR_CUDA;
  return spec_attrs<T, 8>() || spec_attrs<T, 19>() ? MLS6_ERR_CUDA : MLS6_OK;
}
template int prepare_spectral<float>(Plan*);
template int prepare_spectral<double>(Plan*);

template <typename T, int MAXR>
static void launch_spec(Plan* p, const SpecArgs<T>& A, bool vir, unsigned ch, cudaStream_t st) {
  const size_t pl = spec_plane_smem<T>(A.n[0], A.n[1], A.pitch), z = spec_z_smem<T>(A.n[2]);
  const dim3 zg((unsigned)cdiv(A.RL, kSpecCols), ch), planes(A.n[2], ch);
  // a block of a small plane only as large as its work
  const int th = (int)std::min((long)spec_plane_threads<T, MAXR>(),
                               std::max(128L, cdiv(cdiv((long)A.RL, 4), 32) * 32));
  launch_pdl(k_spec_fwd<T, MAXR>, planes, th, pl, st, A);
  launch_pdl(k_spec_z<T, MAXR>, zg, kSpecThreads, z, st, A, T(1));
  launch_pdl(vir ? k_spec_tree<T, true> : k_spec_tree<T, false>,
             dim3((unsigned)p->lv[p->levels].np, ch), kSpecThreads, spec_tree_smem<T>(A.l), st, A);
  launch_pdl(k_spec_z<T, MAXR>, zg, kSpecThreads, z, st, A, T(-1));
  launch_pdl(k_spec_inv<T, MAXR>, planes, th, pl, st, A);
}

template <typename T> int launch_spectral(Plan* p, bool vir, bool lb, cudaStream_t st) {
  const SpecArgs<T> A = spec_args<T>(p, lb);
  unsigned long long r = 0;  // a radix above 8 on any axis
  for (int d = 0; d < 3; ++d)
    for (unsigned long long q = p->spec_rad[d]; q; q >>= 5) r = std::max(r, q & 31);
  if (r > 8)
    launch_spec<T, 19>(p, A, vir, lb ? 7 : 1, st);
  else
    launch_spec<T, 8>(p, A, vir, lb ? 7 : 1, st);
  return 5;
}
template int launch_spectral<float>(Plan*, bool, bool, cudaStream_t);
template int launch_spectral<double>(Plan*, bool, bool, cudaStream_t);

#endif  // MLS6_DEVICE_ONLY
}  // namespace mls6
