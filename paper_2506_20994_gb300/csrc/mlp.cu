// Learned element preconditioner: a two-layer perceptron per element,
//   x = (minv .* r)_e / s_e,  h = tanh(x W1 + b1),  y = h W2 + b2,
// whose output, scaled back by s_e, is added to the Jacobi step (see the
// flexible CG in cg.cu).  The paper has no learned component; this follows
// the project's learned-preconditioner workload.
//
// * Apply (inference): both layers are small dense GEMMs over a tile of 64
//   elements, run on the tensor cores with bf16 operands and fp32
//   accumulation (mma.sync m16n8k16); x is staged in shared memory chunk by
//   chunk, the hidden layer stays in shared memory, and the output goes
//   through shared memory in 128-column slabs so that every global access
//   is a coalesced row segment.
// * Training: fp32 SIMT kernels with a fixed summation order (deterministic,
//   no atomics): forward, mean-squared loss, backpropagation, Adam (Kingma &
//   Ba 2015).  The products are small (25 million multiply-adds at 512 rows,
//   lx = 8, 48 hidden units: under a microsecond of arithmetic), so they are
//   cut for latency: see skinny_kernel.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "alloc.h"
#include "common.cuh"
#include "df64.cuh"
#include "mlp.cuh"
#include "reduce.cuh"

namespace {

constexpr int kTE = 64;     // elements per inference block
constexpr int kKC = 64;     // k-chunk of the first layer
constexpr int kThreads = 256;

inline int round_up(int a, int b) { return (a + b - 1) / b * b; }

// fp32 -> fp64 bits without the fp64 pipe: normal numbers exactly, Inf and
// NaN to Inf and NaN, subnormals and zero to signed zero.
AX_D double f2d(float f) {
  const uint32_t b = __float_as_uint(f);
  const uint32_t e = (b >> 23) & 0xFFu;
  uint64_t d = ((uint64_t)(b & 0x80000000u) << 32);
  if (e == 0xFFu)
    d |= (0x7FFull << 52) | ((uint64_t)(b & 0x7FFFFFu) << 29);
  else if (e != 0u)
    d |= ((uint64_t)(e + 896u) << 52) | ((uint64_t)(b & 0x7FFFFFu) << 29);
  return __longlong_as_double((long long)d);
}
AX_D float to_f32(double x) { return ax::df::split(x).hi; }
AX_D float to_f32(float x) { return x; }
template <typename T>
AX_D T from_f32(float y);
template <>
AX_D double from_f32<double>(float y) { return f2d(y); }
template <>
AX_D float from_f32<float>(float y) { return y; }

AX_D uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);  // .x = lo (low half)
  return *reinterpret_cast<uint32_t *>(&v);
}

AX_D void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
      "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Inference over a tile of kTE elements.  Weights (bf16, padded with
// zeros): W1T [HP][NP] (k contiguous per hidden unit), b1 [HP] (fp32),
// W2T [NP][HP] (k contiguous per output), b2 [NP] (fp32).
// Global memory is touched only by coalesced row-contiguous passes: the
// input chunk is loaded one row segment per warp into xs, and each 128-wide
// output slab goes through ys before it is scaled and stored.
// Shared memory: xs [kTE][kKC+8] bf16, hs [kTE][HP+8] bf16,
// ys [kTE][kYC+4] fp32, s [kTE] fp32, s_part [kTE][2] fp32.
constexpr int kYC = 128;  // output columns per epilogue slab

inline size_t apply_smem(int HP) {
  return (size_t)kTE * (kKC + 8) * 2 + (size_t)kTE * (HP + 8) * 2 + (size_t)kTE * (kYC + 4) * 4 +
         (size_t)kTE * 3 * 4;
}

template <typename T, bool SYM>
__global__ void __launch_bounds__(kThreads)
mlp_apply_kernel(T *__restrict__ corr, const T *__restrict__ r, const T *__restrict__ minv,
                 const T *__restrict__ mask, const T *__restrict__ cw,
                 const float *__restrict__ sc, const __nv_bfloat16 *__restrict__ W1T,
                 const float *__restrict__ b1, const __nv_bfloat16 *__restrict__ W2T,
                 const float *__restrict__ b2, int N, int NP, int HP, int nelv) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int XS = kKC + 8, HS = HP + 8, YS = kYC + 4;  // row strides, padded
  __nv_bfloat16 *xs = reinterpret_cast<__nv_bfloat16 *>(smem_raw);
  __nv_bfloat16 *hs = xs + kTE * XS;
  float *ys = reinterpret_cast<float *>(hs + kTE * HS);
  float *s_sh = ys + kTE * YS;
  float *s_part = s_sh + kTE;  // [kTE][2]

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t4 = lane & 3;
  const long long e0 = (long long)blockIdx.x * kTE;
  // input scale of the residual and activation of the hidden layer; the
  // symmetric form is linear, so its per-element normalisation cancels and
  // is skipped, and its scale sqrt(minv) comes precomputed in sc if given
  auto in_scale = [&](size_t q) {
    return SYM ? (sc ? sc[q] : sqrtf(to_f32(minv[q]))) : to_f32(minv[q]);
  };
  auto act = [](float a) { return SYM ? a : tanhf(a); };
  const int nel = (int)min((long long)kTE, nelv - e0);

  // ---- layer 1: acc = x W1 over k chunks (and ||x||^2 per row, tanh form)
  const int mt = warp & 3;        // rows mt*16 .. +15
  const int nh = warp >> 2;       // n-tiles nh, nh+2, ...
  const int n_tiles1 = HP / 8;
  float acc1[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc1[a][b] = 0.f;
  const int lcol = tid & 63;      // loader: column of the chunk
  const int lrow0 = tid >> 6;     // loader: rows lrow0 + 4 i
  float ss[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) ss[i] = 0.f;
  for (int kc = 0; kc < NP; kc += kKC) {
    __syncthreads();
    const int k = kc + lcol;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int row = lrow0 + 4 * i;
      float v = 0.f;
      if (row < nel && k < N) {
        const size_t q = (size_t)(e0 + row) * N + k;
        v = in_scale(q) * to_f32(r[q]);
      }
      if (!SYM) ss[i] = fmaf(v, v, ss[i]);
      xs[row * XS + lcol] = __float2bfloat16_rn(v);
    }
    __syncthreads();
    const int kmax = min(kKC, NP - kc);
#pragma unroll
    for (int ks = 0; ks < kKC; ks += 16) {
      if (ks >= kmax) break;
      uint32_t a[4];
      const __nv_bfloat16 *x0 = xs + (mt * 16 + g) * XS + ks + 2 * t4;
      const __nv_bfloat16 *x1 = x0 + 8 * XS;
      a[0] = *reinterpret_cast<const uint32_t *>(x0);
      a[1] = *reinterpret_cast<const uint32_t *>(x1);
      a[2] = *reinterpret_cast<const uint32_t *>(x0 + 8);
      a[3] = *reinterpret_cast<const uint32_t *>(x1 + 8);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int nt = nh + 2 * j;
        if (nt < n_tiles1) {
          const __nv_bfloat16 *w = W1T + (size_t)(nt * 8 + g) * NP + kc + ks + 2 * t4;
          const uint32_t b0 = __ldg(reinterpret_cast<const unsigned int *>(w));
          const uint32_t b1r = __ldg(reinterpret_cast<const unsigned int *>(w + 8));
          mma_bf16(acc1[j], a, b0, b1r);
        }
      }
    }
  }
  // row norms: each warp holds 32 columns of its rows; fixed-order sums
  if (!SYM) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      float v = ss[i];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
      if (lane == 0) s_part[(lrow0 + 4 * i) * 2 + (warp & 1)] = v;
    }
  }
  __syncthreads();
  if (tid < kTE) s_sh[tid] = SYM ? 1.f : sqrtf(s_part[2 * tid] + s_part[2 * tid + 1]);
  __syncthreads();
  // hidden layer: h = act(acc / s + b1) -> shared memory (bf16)
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int nt = nh + 2 * j;
    if (nt < n_tiles1) {
      const int col = nt * 8 + 2 * t4;
      const int r0 = mt * 16 + g, r1 = r0 + 8;
      const float i0 = s_sh[r0] > 0.f ? 1.f / s_sh[r0] : 0.f;
      const float i1 = s_sh[r1] > 0.f ? 1.f / s_sh[r1] : 0.f;
      const float bb0 = b1[col], bb1 = b1[col + 1];
      *reinterpret_cast<uint32_t *>(&hs[r0 * HS + col]) =
          pack_bf16(act(acc1[j][0] * i0 + bb0), act(acc1[j][1] * i0 + bb1));
      *reinterpret_cast<uint32_t *>(&hs[r1 * HS + col]) =
          pack_bf16(act(acc1[j][2] * i1 + bb0), act(acc1[j][3] * i1 + bb1));
    }
  }
  __syncthreads();

  // ---- layer 2: y = h W2 + b2 in slabs of kYC outputs, epilogue
  // corr = mask * c * s * y (tanh form) or sqrt(minv) * y (symmetric form)
  const int half = warp >> 2;
  const int n_tiles2 = NP / 8;
  const int r0 = mt * 16 + g, r1 = r0 + 8;
  const int ocol = tid & (kYC - 1), orow0 = tid / kYC;  // epilogue mapping
  for (int nb0 = 0; nb0 < n_tiles2; nb0 += kYC / 8) {
    float acc2[8][4];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc2[a][b] = 0.f;
#pragma unroll
    for (int ks = 0; ks < 64; ks += 16) {  // HP <= 64
      if (ks >= HP) break;
      uint32_t a[4];
      const __nv_bfloat16 *h0 = hs + r0 * HS + ks + 2 * t4;
      const __nv_bfloat16 *h1 = hs + r1 * HS + ks + 2 * t4;
      a[0] = *reinterpret_cast<const uint32_t *>(h0);
      a[1] = *reinterpret_cast<const uint32_t *>(h1);
      a[2] = *reinterpret_cast<const uint32_t *>(h0 + 8);
      a[3] = *reinterpret_cast<const uint32_t *>(h1 + 8);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int nt = nb0 + half * 8 + j;
        if (nt < n_tiles2) {
          const __nv_bfloat16 *w = W2T + (size_t)(nt * 8 + g) * HP + ks + 2 * t4;
          const uint32_t b0 = __ldg(reinterpret_cast<const unsigned int *>(w));
          const uint32_t b1r = __ldg(reinterpret_cast<const unsigned int *>(w + 8));
          mma_bf16(acc2[j], a, b0, b1r);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int col = (half * 8 + j) * 8 + 2 * t4;  // within the slab
      *reinterpret_cast<float2 *>(&ys[r0 * YS + col]) = make_float2(acc2[j][0], acc2[j][1]);
      *reinterpret_cast<float2 *>(&ys[r1 * YS + col]) = make_float2(acc2[j][2], acc2[j][3]);
    }
    __syncthreads();
    const int o = nb0 * 8 + ocol;
    if (o < N) {
      const float bo = b2[o];
      // fixed trip count, unrolled: the loads of several rows are in flight
      // together instead of one latency per row
#pragma unroll 8
      for (int j = 0; j < kTE / (kThreads / kYC); ++j) {
        const int row = orow0 + j * (kThreads / kYC);
        if (row < nel) {
          const size_t q = (size_t)(e0 + row) * N + o;
          const float y = ys[row * YS + ocol] + bo;
          const float osc = SYM ? in_scale(q) : to_f32(mask[q]) * to_f32(cw[q]);
          corr[q] = from_f32<T>(osc * s_sh[row] * y);
        }
      }
    }
    __syncthreads();
  }
}

// Symmetric form with its scale precomputed (sc = sqrt(minv), fp32) and an
// even number of points per element: a block takes 16 elements (the rows of
// the mma tiles) through both layers.  All the warps load and scale the rows
// together (every load of a row in flight at once) into shared memory as
// bf16; the warps then share layer 1's hidden n-tiles and, from the hidden
// layer in shared memory, layer 2's output tiles.  Weights come through L1/L2.
// Rows of shared memory are padded by 8 values, so that the fragment loads
// (8 rows x 4 words) touch every bank once.
// With one warp streaming 16 elements by itself, 4096 elements were 256 warps
// on 152 SMs, each a chain of 32 load latencies: 42 us, against 24 us here
// (fp32, lx = 8, 48 hidden units) with four warps.  Eight shorten the chain of
// each warp again: a refinement iteration with the network (lx = 8) takes 84.8
// against 93.9 us at 16^3 elements, 40.8 / 45.3 at 6^3, 268 / 273 at 26^3;
// sixteen 83.2 at 16^3 but 277 at 26^3.  Sums keep their order (k ascending in
// each tile), so the results are the same bits.
constexpr int kSymWarps = 8;  // warps per block

template <typename T>
struct Pair;  // two consecutive values of T
template <>
struct Pair<double> {
  using V = double2;
};
template <>
struct Pair<float> {
  using V = float2;
};

template <int NT1>
inline size_t sym_smem(int NP) {
  return (size_t)16 * (NP + 8) * 2 + (size_t)16 * (NT1 * 8 + 8) * 2;
}

template <typename T, int NT1>  // NT1 = HP / 8 hidden n-tiles
__global__ void __launch_bounds__(kSymWarps * 32)
mlp_sym_apply_kernel(T *__restrict__ corr, const T *__restrict__ r,
                     const float *__restrict__ sc, const __nv_bfloat16 *__restrict__ W1T,
                     const __nv_bfloat16 *__restrict__ W2T, int N, int NP, int nelv) {
  using V = typename Pair<T>::V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int HP = NT1 * 8, HS = HP + 8;
  const int XS = NP + 8;
  __nv_bfloat16 *xs = reinterpret_cast<__nv_bfloat16 *>(smem_raw);
  __nv_bfloat16 *hs = xs + 16 * XS;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, g = lane >> 2, t4 = lane & 3;
  const long long e0 = (long long)blockIdx.x * 16;
  const int nel = (int)min(16ll, (long long)nelv - e0);

  ax::grid_wait();
  ax::grid_go();
  // the scaled rows, warp w rows w, w + kSymWarps (N even: pairs stay in a row)
  for (int row = wp; row < 16; row += kSymWarps) {
    const size_t base = (size_t)(e0 + (row < nel ? row : 0)) * N;
#pragma unroll 8
    for (int k = 2 * lane; k < NP; k += 64) {
      uint32_t x = 0u;
      if (row < nel && k < N) {
        const V rv = __ldcg(reinterpret_cast<const V *>(r + base + k));
        const float2 sv = __ldcg(reinterpret_cast<const float2 *>(sc + base + k));
        x = pack_bf16(sv.x * to_f32(rv.x), sv.y * to_f32(rv.y));
      }
      *reinterpret_cast<uint32_t *>(xs + row * XS + k) = x;
    }
  }
  __syncthreads();

  // layer 1: hidden n-tiles wp, wp + kSymWarps
  const __nv_bfloat16 *x0 = xs + g * XS + 2 * t4, *x1 = x0 + 8 * XS;
  constexpr int TW = (NT1 + kSymWarps - 1) / kSymWarps;
  float acc[TW][4];
#pragma unroll
  for (int j = 0; j < TW; ++j)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[j][q] = 0.f;
#pragma unroll 4
  for (int ks = 0; ks < NP; ks += 16) {
    const uint32_t a[4] = {*reinterpret_cast<const uint32_t *>(x0 + ks),
                           *reinterpret_cast<const uint32_t *>(x1 + ks),
                           *reinterpret_cast<const uint32_t *>(x0 + ks + 8),
                           *reinterpret_cast<const uint32_t *>(x1 + ks + 8)};
#pragma unroll
    for (int j = 0; j < TW; ++j) {
      const int nt = wp + j * kSymWarps;
      if (nt < NT1) {  // warp-uniform
        const __nv_bfloat16 *w = W1T + (size_t)(nt * 8 + g) * NP + ks + 2 * t4;
        mma_bf16(acc[j], a, __ldg(reinterpret_cast<const unsigned int *>(w)),
                 __ldg(reinterpret_cast<const unsigned int *>(w + 8)));
      }
    }
  }
#pragma unroll
  for (int j = 0; j < TW; ++j) {
    const int nt = wp + j * kSymWarps;
    if (nt < NT1) {
      *reinterpret_cast<uint32_t *>(hs + g * HS + nt * 8 + 2 * t4) = pack_bf16(acc[j][0], acc[j][1]);
      *reinterpret_cast<uint32_t *>(hs + (g + 8) * HS + nt * 8 + 2 * t4) =
          pack_bf16(acc[j][2], acc[j][3]);
    }
  }
  __syncthreads();

  // layer 2: output tiles wp, wp + kSymWarps, ...; corr = sc * y
  uint32_t a2[NT1 / 2][4];
#pragma unroll
  for (int q = 0; q < NT1 / 2; ++q) {
    const __nv_bfloat16 *h0 = hs + g * HS + 16 * q + 2 * t4, *h1 = h0 + 8 * HS;
    a2[q][0] = *reinterpret_cast<const uint32_t *>(h0);
    a2[q][1] = *reinterpret_cast<const uint32_t *>(h1);
    a2[q][2] = *reinterpret_cast<const uint32_t *>(h0 + 8);
    a2[q][3] = *reinterpret_cast<const uint32_t *>(h1 + 8);
  }
  const bool ok0 = g < nel, ok1 = g + 8 < nel;
  const size_t row0 = (size_t)(e0 + (ok0 ? g : 0)) * N, row1 = (size_t)(e0 + (ok1 ? g + 8 : 0)) * N;
#pragma unroll 4
  for (int nt = wp; nt < NP / 8; nt += kSymWarps) {
    const int col = nt * 8 + 2 * t4;
    const bool in = col < N;
    const float2 zero = make_float2(0.f, 0.f);
    const float2 s0 = in && ok0 ? __ldcg(reinterpret_cast<const float2 *>(sc + row0 + col)) : zero;
    const float2 s1 = in && ok1 ? __ldcg(reinterpret_cast<const float2 *>(sc + row1 + col)) : zero;
    float acc2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int q = 0; q < NT1 / 2; ++q) {
      const __nv_bfloat16 *w = W2T + (size_t)(nt * 8 + g) * HP + 16 * q + 2 * t4;
      mma_bf16(acc2, a2[q], __ldg(reinterpret_cast<const unsigned int *>(w)),
               __ldg(reinterpret_cast<const unsigned int *>(w + 8)));
    }
    if (in && ok0) {
      V o;
      o.x = from_f32<T>(s0.x * acc2[0]);
      o.y = from_f32<T>(s0.y * acc2[1]);
      *reinterpret_cast<V *>(corr + row0 + col) = o;
    }
    if (in && ok1) {
      V o;
      o.x = from_f32<T>(s1.x * acc2[2]);
      o.y = from_f32<T>(s1.y * acc2[3]);
      *reinterpret_cast<V *>(corr + row1 + col) = o;
    }
  }
}

template <typename T, int NT1>
int sym_apply(T *corr, const T *r, const float *sc, const __nv_bfloat16 *w1,
              const __nv_bfloat16 *w2, int N, int NP, int nelv, cudaStream_t st) {
  auto kern = mlp_sym_apply_kernel<T, NT1>;
  const size_t smem = sym_smem<NT1>(NP);
  static std::atomic<size_t> granted[ax::kMaxDevices];
  if (!ax::grant_smem(kern, smem, granted)) return AX_EINVAL;
  // not chained: the few blocks of a small mesh would crowd onto the SMs that
  // the kernel in front leaves first
  return ax::launch_chained(false, kern, (unsigned)((nelv + 15) / 16), kSymWarps * 32, smem, st, corr,
                            r, sc, w1, w2, N, NP, nelv);
}

// ---------------------------------------------------------------- training
// X[b][k] = (minv r)_e / s, T[b][k] = (err - minv r)_e / s for e = idx[b]
__global__ void gather_pairs_kernel(float *__restrict__ X, float *__restrict__ Tt,
                                    const double *__restrict__ r, const double *__restrict__ err,
                                    const double *__restrict__ minv, const int *__restrict__ idx,
                                    int N) {
  const int b = blockIdx.x;
  const size_t base = (size_t)idx[b] * N;
  double ss = 0.0;
  for (int k = threadIdx.x; k < N; k += blockDim.x) {
    const double z = minv[base + k] * r[base + k];
    ss += z * z;
  }
  double v[1] = {ss};
  ax::block_sum<1>(v);
  __shared__ double s_b;
  if (threadIdx.x == 0) s_b = sqrt(v[0]);
  __syncthreads();
  const double inv = s_b > 0.0 ? 1.0 / s_b : 0.0;
  for (int k = threadIdx.x; k < N; k += blockDim.x) {
    const double z = minv[base + k] * r[base + k];
    X[(size_t)b * N + k] = (float)(z * inv);
    Tt[(size_t)b * N + k] = (float)((err[base + k] - z) * inv);
  }
}

// C[m][h] = sum_k A(m, k) B(k, h), h < Hd <= 64: the products of training
// whose one side is the hidden layer.  A block takes kRows rows of C and walks
// k in chunks of kChunk: A's and B's chunk are staged in shared memory while
// the next one's loads are in flight in registers, and four groups of 64
// threads (thread (slice, h)) take a quarter of the chunk each; their sums are
// added in a fixed order.  One thread per output with a chain over all of k
// left 96 blocks each waiting on 512 dependent loads (the four products of a
// training step took over 200 of its 415 us at 512 rows, lx = 8, 48 hidden
// units); the slices alone, with B read from L2 inside the chain, 19-32 us a
// product; staged, 7-11 us (GB300, cold).
// AT: A stored [k][m], else [m][k].  BT: B stored [h][k], else [k][h] with
// ldb = Hd (one contiguous 16-byte aligned run per chunk).  ONES: row M - 1
// of A is all ones (the bias gradient).  A second pair (A2, B2) with the same
// shapes, if given, continues the same sums.  epi(m, h, sum) receives each
// output once; csum(m, sum_k A(m, k)) each row's sum (the output-bias
// gradient) when CSUM.
constexpr int kRows = 4, kSlices = 4, kChunk = 128;

template <bool AT, bool BT, bool ONES, bool CSUM, class Epi, class Csum>
__global__ void __launch_bounds__(kThreads)
skinny_kernel(const float *__restrict__ A, const float *__restrict__ B,
              const float *__restrict__ A2, const float *__restrict__ B2, int M, int K, int Hd,
              int lda, int ldb, Epi epi, Csum csum) {
  constexpr int NA = kRows * kChunk / kThreads;       // A values a thread stages
  constexpr int NB = kChunk * 64 / 4 / kThreads;      // B float4 a thread stages (Hd = 64)
  constexpr int PB = 65;                              // padded row of a transposed B
  __shared__ float4 As[kChunk];
  __shared__ float4 Bs4[(kChunk * PB + 3) / 4];
  __shared__ float red[kSlices][kRows][64];
  __shared__ float redc[kSlices][kRows];
  float *Bs = reinterpret_cast<float *>(Bs4);
  const int tid = threadIdx.x, h = tid & 63, sl = tid >> 6;
  const int m0 = blockIdx.x * kRows;
  const int Mr = ONES ? M - 1 : M;  // rows that A stores
  const int BS = BT ? PB : Hd;      // row stride of Bs
  float acc[kRows] = {0.f, 0.f, 0.f, 0.f}, cs[kRows] = {0.f, 0.f, 0.f, 0.f};
  const int chunks = (K + kChunk - 1) / kChunk, steps = A2 ? 2 * chunks : chunks;
  float ra[NA];
  float4 rb[NB];
  // one step's values into registers
  auto load = [&](int step) {
    const bool second = step >= chunks;
    const float *a = second ? A2 : A, *b = second ? B2 : B;
    const int k0 = (second ? step - chunks : step) * kChunk;
    const int kn = min(kChunk, K - k0);
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int v = tid + q * kThreads;
      const int r = AT ? v % kRows : v / kChunk, k = AT ? v / kRows : v % kChunk;
      const int m = m0 + r;
      ra[q] = k >= kn ? 0.f
              : m < Mr ? __ldcg(AT ? a + (size_t)(k0 + k) * lda + m : a + (size_t)m * lda + k0 + k)
              : ONES && m == Mr ? 1.f : 0.f;
    }
    const int nv = kn * Hd;
    if constexpr (BT) {
#pragma unroll
      for (int q = 0; q < 4 * NB; ++q) {  // value (row v / kChunk of B, k = v % kChunk)
        const int v = tid + q * kThreads, hh = v / kChunk, k = v % kChunk;
        reinterpret_cast<float *>(rb)[q] =
            hh < Hd && k < kn ? __ldcg(b + (size_t)hh * ldb + k0 + k) : 0.f;
      }
    } else {
      const float *src = b + (size_t)k0 * Hd;
#pragma unroll
      for (int q = 0; q < NB; ++q) {
        const int v = 4 * (tid + q * kThreads);
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (v + 3 < nv) {
          x = __ldcg(reinterpret_cast<const float4 *>(src + v));
        } else {
          if (v < nv) x.x = __ldcg(src + v);
          if (v + 1 < nv) x.y = __ldcg(src + v + 1);
          if (v + 2 < nv) x.z = __ldcg(src + v + 2);
        }
        rb[q] = x;
      }
    }
  };
  ax::grid_wait();
  ax::grid_go();
  load(0);
  for (int step = 0; step < steps; ++step) {
    if (step) __syncthreads();
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int v = tid + q * kThreads;
      const int r = AT ? v % kRows : v / kChunk, k = AT ? v / kRows : v % kChunk;
      reinterpret_cast<float *>(As)[k * kRows + r] = ra[q];
    }
    if constexpr (BT) {
#pragma unroll
      for (int q = 0; q < 4 * NB; ++q) {
        const int v = tid + q * kThreads;
        Bs[(v % kChunk) * PB + v / kChunk] = reinterpret_cast<const float *>(rb)[q];
      }
    } else {
#pragma unroll
      for (int q = 0; q < NB; ++q) Bs4[tid + q * kThreads] = rb[q];
    }
    __syncthreads();
    if (step + 1 < steps) load(step + 1);
    if (h < Hd) {
      const int ka = sl * (kChunk / kSlices);
#pragma unroll 8
      for (int k = ka; k < ka + kChunk / kSlices; ++k) {  // zeros past the end of k
        const float bv = Bs[k * BS + h];
        const float4 av = As[k];
        acc[0] = fmaf(av.x, bv, acc[0]);
        acc[1] = fmaf(av.y, bv, acc[1]);
        acc[2] = fmaf(av.z, bv, acc[2]);
        acc[3] = fmaf(av.w, bv, acc[3]);
        if (CSUM) {
          cs[0] += av.x;
          cs[1] += av.y;
          cs[2] += av.z;
          cs[3] += av.w;
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    red[sl][r][h] = acc[r];
    if (CSUM && h == 0) redc[sl][r] = cs[r];
  }
  __syncthreads();
  const int r = sl;  // four slices, four rows: thread (slice, h) finishes row `slice`
  if (m0 + r < M && h < Hd)
    epi(m0 + r, h, (red[0][r][h] + red[1][r][h]) + (red[2][r][h] + red[3][r][h]));
  if (CSUM && h == 0 && m0 + r < M)
    csum(m0 + r, (redc[0][r] + redc[1][r]) + (redc[2][r] + redc[3][r]));
}

struct NoCsum {
  AX_D void operator()(int, float) const {}
};
// H = act(sum + b1)
struct EpiHidden {
  float *H;
  const float *b1;
  int Hd, sym;
  AX_D void operator()(int b, int h, float a) const {
    const float v = a + __ldcg(b1 + h);
    H[(size_t)b * Hd + h] = sym ? v : tanhf(v);
  }
};
// dP = sum (1 - H^2) (the symmetric form is linear)
struct EpiBack {
  float *dP;
  const float *H;
  int Hd, sym;
  AX_D void operator()(int b, int h, float a) const {
    const size_t q = (size_t)b * Hd + h;
    const float hv = __ldcg(H + q);
    dP[q] = sym ? a : a * (1.f - hv * hv);
  }
};
// row-major [m][h] (W1's gradient; row N is b1's)
struct EpiRows {
  float *g;
  int Hd;
  AX_D void operator()(int m, int h, float a) const { g[(size_t)m * Hd + h] = a; }
};
// transposed [h][m] (W2's gradient), and its bias
struct EpiCols {
  float *g;
  int N;
  AX_D void operator()(int m, int h, float a) const { g[(size_t)h * N + m] = a; }
};
struct CsumBias {
  float *g;
  AX_D void operator()(int m, float a) const { g[m] = a; }
};

// Y(b, o) = sum_h H[b][h] W2[h][o] + b2[o] for kRows rows and 256 outputs a
// block; fin(b, o, y) receives each.
template <class Fin>
AX_D void out_rows(const float *__restrict__ H, const float *__restrict__ theta, int B, int N,
                   int Hd, Fin fin) {
  __shared__ float4 Hs[64];
  ax::grid_wait();
  ax::grid_go();
  const int b0 = blockIdx.x * kRows, o = blockIdx.y * kThreads + threadIdx.x;
  const float *W2 = theta + (size_t)N * Hd + Hd, *b2 = W2 + (size_t)Hd * N;
  if (threadIdx.x < Hd * kRows) {
    const int r = threadIdx.x / Hd, h = threadIdx.x % Hd;
    reinterpret_cast<float *>(Hs)[h * kRows + r] =
        b0 + r < B ? __ldcg(H + (size_t)(b0 + r) * Hd + h) : 0.f;
  }
  __syncthreads();
  if (o >= N) return;
  float acc[kRows] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
  for (int h = 0; h < Hd; ++h) {
    const float w = __ldcg(W2 + (size_t)h * N + o);
    const float4 v = Hs[h];
    acc[0] = fmaf(v.x, w, acc[0]);
    acc[1] = fmaf(v.y, w, acc[1]);
    acc[2] = fmaf(v.z, w, acc[2]);
    acc[3] = fmaf(v.w, w, acc[3]);
  }
  const float bo = __ldcg(b2 + o);
#pragma unroll
  for (int r = 0; r < kRows; ++r)
    if (b0 + r < B) fin(b0 + r, o, acc[r] + bo);
}

// Y = H W2 + b2; dY = 2 (Y - T) / (B N); per-block partial of sum (Y-T)^2
__global__ void __launch_bounds__(kThreads)
fwd_out_loss_kernel(float *__restrict__ Y, float *__restrict__ dY, const float *__restrict__ H,
                    const float *__restrict__ Tt, const float *__restrict__ theta, int B, int N,
                    int Hd, double *__restrict__ partials) {
  double l = 0.0;
  out_rows(H, theta, B, N, Hd, [&](int b, int o, float y) {
    const size_t q = (size_t)b * N + o;
    Y[q] = y;
    const float res = y - __ldcg(Tt + q);
    dY[q] = 2.f * res / ((float)B * (float)N);
    l += (double)res * (double)res;
  });
  double v[1] = {l};
  ax::block_sum<1>(v);
  if (threadIdx.x == 0) partials[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = v[0];
}

// The energy-norm training's forward: corr = osc[q] s_b Y(b, o) (fp64), the
// element's scaled output before assembly
__global__ void __launch_bounds__(kThreads)
fwd_out_corr_kernel(double *__restrict__ corr, const float *__restrict__ H,
                    const float *__restrict__ theta, const double *__restrict__ osc,
                    const double *__restrict__ s, int B, int N, int Hd) {
  out_rows(H, theta, B, N, Hd, [&](int b, int o, float y) {
    const size_t q = (size_t)b * N + o;
    corr[q] = __ldcg(osc + q) * __ldcg(s + b) * (double)y;
  });
}

__global__ void adam_kernel(float *__restrict__ theta, float *__restrict__ m,
                            float *__restrict__ v, const float *__restrict__ g, int64_t n,
                            float lr, float b1, float b2, float eps, float c1, float c2) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  const float gq = g[q];
  const float mq = b1 * m[q] + (1.f - b1) * gq;
  const float vq = b2 * v[q] + (1.f - b2) * gq * gq;
  m[q] = mq;
  v[q] = vq;
  theta[q] -= lr * (mq / c1) / (sqrtf(vq / c2) + eps);
}

// Adam of the symmetric form: the free parameters are W1 (W2 = W1^T, zero
// biases); each thread updates one and writes its mirror image
__global__ void adam_sym_kernel(float *__restrict__ theta, float *__restrict__ m,
                                float *__restrict__ v, const float *__restrict__ g, int N, int Hd,
                                float lr, float b1, float b2, float eps, float c1, float c2) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  ax::grid_wait();  // every thread, also one without a parameter
  ax::grid_go();
  if (q >= (int64_t)N * Hd) return;
  const float gq = __ldcg(g + q);
  const float mq = b1 * __ldcg(m + q) + (1.f - b1) * gq;
  const float vq = b2 * __ldcg(v + q) + (1.f - b2) * gq * gq;
  m[q] = mq;
  v[q] = vq;
  const float t = __ldcg(theta + q) - lr * (mq / c1) / (sqrtf(vq / c2) + eps);
  theta[q] = t;
  theta[(size_t)N * Hd + Hd + (size_t)(q % Hd) * N + q / Hd] = t;
}

// bf16 inference copy: W1T [HP][NP], b1 [HP] (fp32), W2T [NP][HP], b2 [NP] (fp32)
__global__ void refresh_bf16_kernel(__nv_bfloat16 *__restrict__ W1T, float *__restrict__ b1p,
                                    __nv_bfloat16 *__restrict__ W2T, float *__restrict__ b2p,
                                    const float *__restrict__ theta, int N, int Hd, int NP,
                                    int HP) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const float *W1 = theta, *b1 = theta + (size_t)N * Hd;
  const float *W2 = b1 + Hd, *b2 = W2 + (size_t)Hd * N;
  const int64_t n1 = (int64_t)HP * NP;
  if (q < n1) {
    const int h = (int)(q / NP), k = (int)(q % NP);
    W1T[q] = __float2bfloat16_rn((h < Hd && k < N) ? W1[(size_t)k * Hd + h] : 0.f);
  }
  if (q < (int64_t)NP * HP) {
    const int o = (int)(q / HP), h = (int)(q % HP);
    W2T[q] = __float2bfloat16_rn((h < Hd && o < N) ? W2[(size_t)h * N + o] : 0.f);
  }
  if (q < HP) b1p[q] = q < Hd ? b1[q] : 0.f;
  if (q < NP) b2p[q] = q < N ? b2[q] : 0.f;
}

struct Layout {
  int NP, HP;
  size_t w1t, b1p, w2t, b2p;  // offsets (bytes) in theta_bf's allocation
  size_t bytes;
};

Layout layout(const ax_mlp *M) {
  Layout L;
  L.NP = round_up(M->n_in, 16);
  L.HP = round_up(M->n_hid, 16);
  L.w1t = 0;
  L.b1p = L.w1t + (size_t)L.HP * L.NP * 2;
  L.w2t = L.b1p + (size_t)L.HP * 4;
  L.b2p = L.w2t + (size_t)L.NP * L.HP * 2;
  L.bytes = L.b2p + (size_t)L.NP * 4;
  return L;
}

int refresh_bf16(ax_mlp *M, cudaStream_t st) {
  const Layout L = layout(M);
  char *base = reinterpret_cast<char *>(M->theta_bf);
  const int64_t n = std::max<int64_t>((int64_t)L.HP * L.NP, (int64_t)L.NP);
  refresh_bf16_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(
      reinterpret_cast<__nv_bfloat16 *>(base + L.w1t), reinterpret_cast<float *>(base + L.b1p),
      reinterpret_cast<__nv_bfloat16 *>(base + L.w2t), reinterpret_cast<float *>(base + L.b2p),
      M->theta, M->n_in, M->n_hid, L.NP, L.HP);
  return ax::launch_status();
}

inline unsigned blocks_of(int64_t n) { return (unsigned)((n + kThreads - 1) / kThreads); }
inline dim3 out_grid(int B, int N) {
  return dim3((unsigned)((B + kRows - 1) / kRows), (unsigned)((N + kThreads - 1) / kThreads));
}

int ensure_capacity(ax_mlp *M, int B) {
  if (B <= M->cap) return AX_OK;
  M->cap = 0;
  const size_t bn = (size_t)B * M->n_in, bh = (size_t)B * M->n_hid;
  const dim3 og = out_grid(B, M->n_in);
  const size_t nblk = (size_t)og.x * og.y;
  M->Y = nullptr;
  if (int rc = ax::alloc_all({{&M->X, bn}, {&M->T, 2 * bn}, {&M->dY, bn}, {&M->H, bh},
                              {&M->dP, bh}, {&M->es, (size_t)B}, {&M->partials, nblk}}))
    return rc;
  M->Y = M->T + bn;
  M->cap = B;
  return AX_OK;
}

// W2 = W1^T, b1 = b2 = 0
__global__ void tie_params_kernel(float *__restrict__ theta, int N, int Hd) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  float *b1 = theta + (size_t)N * Hd, *W2 = b1 + Hd, *b2 = W2 + (size_t)Hd * N;
  if (q < (int64_t)N * Hd) {
    const int k = (int)(q / Hd), h = (int)(q % Hd);
    W2[(size_t)h * N + k] = theta[q];
  }
  if (q < Hd) b1[q] = 0.f;
  if (q < N) b2[q] = 0.f;
}

// rows perm[b] of the sample set -> the batch buffers
__global__ void gather_rows_kernel(float *__restrict__ X, float *__restrict__ Tt,
                                   const float *__restrict__ Xa, const float *__restrict__ Ta,
                                   const int *__restrict__ perm, int N) {
  const size_t src = (size_t)perm[blockIdx.x] * N, dst = (size_t)blockIdx.x * N;
  for (int k = threadIdx.x; k < N; k += blockDim.x) {
    X[dst + k] = Xa[src + k];
    Tt[dst + k] = Ta[src + k];
  }
}

__global__ void sum_partials_kernel2(const double *__restrict__ p, int n, double *__restrict__ out) {
  ax::warp_sum_partials<1>(p, n, out);
}

template <bool AT, bool BT, bool ONES, bool CSUM, class Epi, class Csum>
int launch_skinny(cudaStream_t st, const float *A, const float *B, const float *A2,
                  const float *B2, int M, int K, int Hd, int lda, int ldb, Epi epi, Csum csum) {
  return ax::launch_chained(true, skinny_kernel<AT, BT, ONES, CSUM, Epi, Csum>,
                            (unsigned)((M + kRows - 1) / kRows), kThreads, 0, st, A, B, A2, B2, M,
                            K, Hd, lda, ldb, epi, csum);
}

// H = act(X W1 + b1)
int launch_hidden(ax_mlp *M, int B, cudaStream_t st) {
  const int N = M->n_in, Hd = M->n_hid;
  const EpiHidden epi{M->H, M->theta + (size_t)N * Hd, Hd, M->arch == AX_MLP_SYM};
  return launch_skinny<false, false, false, false>(st, M->X, M->theta, nullptr, nullptr, B, N, Hd,
                                                   N, Hd, epi, NoCsum{});
}

// Gradient from M->X, M->H, M->dY.  Tanh form: all four blocks.  Symmetric
// form: the gradient of the free parameters W1 (W2's folded in: both are
// [N][Hd] sums over the rows, X^T dP + dY^T H); the rest of M->grad is zero
// from the start and stays so.
int launch_backward(ax_mlp *M, int B, cudaStream_t st) {
  const int N = M->n_in, Hd = M->n_hid;
  const float *none = nullptr;
  if (M->arch == AX_MLP_SYM) {
    // W2 = W1^T, so the back product reads W1's coalesced rows
    if (int rc = launch_skinny<false, false, false, false>(st, M->dY, M->theta, none, none, B, N, Hd,
                                                           N, Hd, EpiBack{M->dP, M->H, Hd, 1},
                                                           NoCsum{}))
      return rc;
    return launch_skinny<true, false, false, false>(st, M->X, M->dP, M->dY, M->H, N, B, Hd, N, Hd,
                                                    EpiRows{M->grad, Hd}, NoCsum{});
  }
  const float *W2 = M->theta + (size_t)N * Hd + Hd;
  float *gW2 = M->grad + (size_t)N * Hd + Hd;
  int rc = launch_skinny<true, false, false, true>(st, M->dY, M->H, none, none, N, B, Hd, N, Hd,
                                                   EpiCols{gW2, N},
                                                   CsumBias{gW2 + (size_t)Hd * N});
  if (rc == AX_OK)
    rc = launch_skinny<false, true, false, false>(st, M->dY, W2, none, none, B, N, Hd, N, N,
                                                  EpiBack{M->dP, M->H, Hd, 0}, NoCsum{});
  if (rc == AX_OK)
    rc = launch_skinny<true, false, true, false>(st, M->X, M->dP, none, none, N + 1, B, Hd, N, Hd,
                                                 EpiRows{M->grad, Hd}, NoCsum{});
  return rc;
}

// forward + loss + gradient on M->X / M->T (B samples)
int loss_grad_dev(ax_mlp *M, int B, cudaStream_t st) {
  const int N = M->n_in, Hd = M->n_hid;
  if (int rc = launch_hidden(M, B, st)) return rc;
  const dim3 og = out_grid(B, N);
  if (ax::launch_chained(true, fwd_out_loss_kernel, og, kThreads, 0, st, M->Y, M->dY, M->H, M->T,
                         M->theta, B, N, Hd, M->partials))
    return AX_ELAUNCH;
  sum_partials_kernel2<<<1, 32, 0, st>>>(M->partials, (int)(og.x * og.y), M->loss_dev);
  return launch_backward(M, B, st);
}

// Adam on M->grad (symmetric form: the tied parameters together)
int adam_dev(ax_mlp *M, float lr, float b1, float b2, float eps, cudaStream_t st) {
  M->adam_step += 1;
  const float c1 = 1.f - powf(b1, (float)M->adam_step);
  const float c2 = 1.f - powf(b2, (float)M->adam_step);
  if (M->arch == AX_MLP_SYM)
    return ax::launch_chained(true, adam_sym_kernel, blocks_of((int64_t)M->n_in * M->n_hid), kThreads,
                              0, st, M->theta, M->m, M->v, M->grad, M->n_in, M->n_hid, lr, b1, b2,
                              eps, c1, c2);
  else
    adam_kernel<<<blocks_of(M->nparam), kThreads, 0, st>>>(M->theta, M->m, M->v, M->grad,
                                                           M->nparam, lr, b1, b2, eps, c1, c2);
  return ax::launch_status();
}

}  // namespace

namespace ax {

int mlp_reserve(ax_mlp *M, int B, int pairs) {
  if (int rc = ensure_capacity(M, B)) return rc;
  if (pairs <= M->kcap) return AX_OK;
  M->kcap = 0;
  if (int rc = alloc_all({{&M->ek, 2 * (size_t)pairs +
                                       (size_t)std::min(pairs, kEnergyPairs) * kRedBlocks}}))
    return rc;
  M->kcap = pairs;
  return AX_OK;
}

// M->X -> H, then corr = osc s_b Y in fp64 (B rows)
int mlp_train_forward_corr(ax_mlp *M, int B, double *corr, const double *osc, const double *s,
                           cudaStream_t st) {
  const int N = M->n_in, Hd = M->n_hid;
  if (int rc = launch_hidden(M, B, st)) return rc;
  return launch_chained(true, fwd_out_corr_kernel, out_grid(B, N), kThreads, 0, st, corr, M->H,
                        M->theta, osc, s, B, N, Hd);
}

// gradient from M->X, M->H and the output gradient M->dY (B rows)
int mlp_train_backward(ax_mlp *M, int B, cudaStream_t st) {
  return launch_backward(M, B, st);
}

int mlp_adam_step(ax_mlp *M, float lr, cudaStream_t st) {
  return adam_dev(M, lr, 0.9f, 0.999f, 1e-8f, st);
}

int mlp_refresh(ax_mlp *M, cudaStream_t st) { return refresh_bf16(M, st); }

int mlp_tie_params(ax_mlp *M, cudaStream_t st) {
  const int N = M->n_in, Hd = M->n_hid;
  const int64_t n = std::max<int64_t>((int64_t)N * Hd, N);
  tie_params_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(M->theta, N, Hd);
  return launch_status();
}

template <typename T>
int mlp_correction(const ax_mlp *M, T *corr, const T *r, const T *minv, const T *mask,
                   const T *c, int nelv, cudaStream_t st, const float *sc) {
  if (nelv <= 0) return AX_OK;
  const Layout L = layout(M);
  const char *base = reinterpret_cast<const char *>(M->theta_bf);
  // the kernel for pairs of values reads and writes r, sc and corr as pairs: a
  // caller's r may start between two (ax_precondition passes it on)
  auto pairs = [](const void *p, size_t size) { return (uintptr_t)p % (2 * size) == 0; };
  if (M->arch == AX_MLP_SYM && sc && M->n_in % 2 == 0 &&
      (L.HP == 16 || L.HP == 32 || L.HP == 48 || L.HP == 64) && pairs(r, sizeof(T)) &&
      pairs(corr, sizeof(T)) && pairs(sc, sizeof(float))) {
    auto w1 = reinterpret_cast<const __nv_bfloat16 *>(base + L.w1t);
    auto w2 = reinterpret_cast<const __nv_bfloat16 *>(base + L.w2t);
    switch (L.HP) {
      case 16: return sym_apply<T, 2>(corr, r, sc, w1, w2, M->n_in, L.NP, nelv, st);
      case 32: return sym_apply<T, 4>(corr, r, sc, w1, w2, M->n_in, L.NP, nelv, st);
      case 48: return sym_apply<T, 6>(corr, r, sc, w1, w2, M->n_in, L.NP, nelv, st);
      default: return sym_apply<T, 8>(corr, r, sc, w1, w2, M->n_in, L.NP, nelv, st);
    }
  }
  const size_t smem = apply_smem(L.HP);
  auto kern = M->arch == AX_MLP_SYM ? mlp_apply_kernel<T, true> : mlp_apply_kernel<T, false>;
  if (smem > 48 * 1024 &&
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
          cudaSuccess) {
    (void)cudaGetLastError();
    return AX_EINVAL;
  }
  const unsigned grid = (unsigned)((nelv + kTE - 1) / kTE);
  kern<<<grid, kThreads, smem, st>>>(
      corr, r, minv, mask, c, sc, reinterpret_cast<const __nv_bfloat16 *>(base + L.w1t),
      reinterpret_cast<const float *>(base + L.b1p),
      reinterpret_cast<const __nv_bfloat16 *>(base + L.w2t),
      reinterpret_cast<const float *>(base + L.b2p), M->n_in, L.NP, L.HP, nelv);
  return launch_status();
}

template int mlp_correction<double>(const ax_mlp *, double *, const double *, const double *,
                                    const double *, const double *, int, cudaStream_t,
                                    const float *);
template int mlp_correction<float>(const ax_mlp *, float *, const float *, const float *,
                                   const float *, const float *, int, cudaStream_t,
                                   const float *);

}  // namespace ax

extern "C" {

int ax_mlp_destroy(ax_mlp *M) {
  if (!M) return AX_OK;
  float *f[] = {M->theta, M->grad, M->m, M->v, M->X, M->T, M->H, M->dY, M->dP};
  for (float *p : f) cudaFree(p);
  cudaFree(M->theta_bf);
  cudaFree(M->partials);
  cudaFree(M->es);
  cudaFree(M->ek);
  cudaFree(M->loss_dev);
  delete M;
  return AX_OK;
}

int ax_mlp_create_ex(ax_mlp **out, int n_in, int n_hid, int arch) {
  if (!out || n_in < 1 || n_in > 4096 || n_hid < 1 || n_hid > 64 ||
      (arch != AX_MLP_TANH && arch != AX_MLP_SYM))
    return AX_EINVAL;
  *out = nullptr;
  ax_mlp *M = new (std::nothrow) ax_mlp();
  if (!M) return AX_ENOMEM;
  M->n_in = n_in;
  M->n_hid = n_hid;
  M->arch = arch;
  M->nparam = (int64_t)n_in * n_hid + n_hid + (int64_t)n_hid * n_in + n_in;
  const Layout L = layout(M);
  const size_t pb = (size_t)M->nparam * 4;
  if (cudaMalloc(&M->theta, pb) != cudaSuccess || cudaMalloc(&M->grad, pb) != cudaSuccess ||
      cudaMalloc(&M->m, pb) != cudaSuccess || cudaMalloc(&M->v, pb) != cudaSuccess ||
      cudaMalloc(&M->theta_bf, L.bytes) != cudaSuccess ||
      cudaMalloc(&M->loss_dev, sizeof(double)) != cudaSuccess ||
      cudaMemset(M->theta, 0, pb) != cudaSuccess || cudaMemset(M->grad, 0, pb) != cudaSuccess ||
      cudaMemset(M->m, 0, pb) != cudaSuccess || cudaMemset(M->v, 0, pb) != cudaSuccess ||
      cudaMemset(M->theta_bf, 0, L.bytes) != cudaSuccess) {
    (void)cudaGetLastError();
    ax_mlp_destroy(M);
    return AX_ENOMEM;
  }
  *out = M;
  return AX_OK;
}

int ax_mlp_create(ax_mlp **out, int n_in, int n_hid) {
  return ax_mlp_create_ex(out, n_in, n_hid, AX_MLP_TANH);
}

int ax_mlp_nparams(const ax_mlp *M, int64_t *n) {
  if (!M || !n) return AX_EINVAL;
  *n = M->nparam;
  return AX_OK;
}

int ax_mlp_set_params(ax_mlp *M, const float *host, int64_t count, void *stream) {
  if (!M || !host || count != M->nparam) return AX_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  if (cudaMemcpyAsync(M->theta, host, count * 4, cudaMemcpyHostToDevice, st) != cudaSuccess ||
      cudaMemsetAsync(M->m, 0, count * 4, st) != cudaSuccess ||
      cudaMemsetAsync(M->v, 0, count * 4, st) != cudaSuccess) {
    (void)cudaGetLastError();
    return AX_ELAUNCH;
  }
  M->adam_step = 0;
  int rc = M->arch == AX_MLP_SYM ? ax::mlp_tie_params(M, st) : AX_OK;
  if (rc == AX_OK) rc = refresh_bf16(M, st);
  if (rc == AX_OK && cudaStreamSynchronize(st) != cudaSuccess) rc = AX_ELAUNCH;
  return rc;
}

int ax_mlp_get_params(const ax_mlp *M, float *host, int64_t count, void *stream) {
  if (!M || !host || count != M->nparam) return AX_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  if (cudaMemcpyAsync(host, M->theta, count * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess) {
    (void)cudaGetLastError();
    return AX_ELAUNCH;
  }
  return AX_OK;
}

int ax_mlp_loss_grad(ax_mlp *M, const float *X, const float *T, int B, double *loss,
                     float *grad_host, void *stream) {
  if (!M || !X || !T || B < 1) return AX_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  int rc = ensure_capacity(M, B);
  if (rc) return rc;
  const size_t bn = (size_t)B * M->n_in * 4;
  if (cudaMemcpyAsync(M->X, X, bn, cudaMemcpyDeviceToDevice, st) != cudaSuccess ||
      cudaMemcpyAsync(M->T, T, bn, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
    return AX_ELAUNCH;
  if ((rc = loss_grad_dev(M, B, st))) return rc;
  double l = 0.0;
  if (cudaMemcpyAsync(&l, M->loss_dev, 8, cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return AX_ELAUNCH;
  if (grad_host && cudaMemcpyAsync(grad_host, M->grad, M->nparam * 4, cudaMemcpyDeviceToHost,
                                   st) != cudaSuccess)
    return AX_ELAUNCH;
  if (cudaStreamSynchronize(st) != cudaSuccess) return AX_ELAUNCH;
  if (loss) *loss = l / ((double)B * M->n_in);
  return AX_OK;
}

int ax_mlp_adam(ax_mlp *M, float lr, float beta1, float beta2, float eps, void *stream) {
  if (!M || !(lr >= 0)) return AX_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  int rc = adam_dev(M, lr, beta1, beta2, eps, st);
  if (rc) return rc;
  return refresh_bf16(M, st);
}

int ax_mlp_forward(const ax_mlp *M, const float *r, const float *minv, const float *mask,
                   const float *c, float *corr, int nelv, void *stream) {
  if (!M || nelv < 0 || (nelv > 0 && !ax::all_nonnull(r, minv, mask, c, corr)))
    return AX_EINVAL;
  return ax::mlp_correction<float>(M, corr, r, minv, mask, c, nelv, (cudaStream_t)stream);
}

int ax_mlp_train(ax_mlp *M, const float *X_all, const float *T_all, int nsamples,
                 const int *perm, int epochs, int batch, float lr, double *final_loss,
                 void *stream) {
  if (!M || !X_all || !T_all || !perm || nsamples < 1 || batch < 1 || epochs < 1 || !(lr > 0))
    return AX_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  batch = std::min(batch, nsamples);
  int rc = ensure_capacity(M, batch);
  if (rc) return rc;
  for (int ep = 0; ep < epochs; ++ep) {
    for (int s0 = 0; s0 + batch <= nsamples; s0 += batch) {
      gather_rows_kernel<<<batch, kThreads, 0, st>>>(M->X, M->T, X_all, T_all,
                                                     perm + (size_t)ep * nsamples + s0, M->n_in);
      if ((rc = loss_grad_dev(M, batch, st))) return rc;
      if ((rc = adam_dev(M, lr, 0.9f, 0.999f, 1e-8f, st))) return rc;
    }
  }
  if ((rc = refresh_bf16(M, st))) return rc;
  double last = 0.0;
  if (cudaMemcpyAsync(&last, M->loss_dev, 8, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return AX_ELAUNCH;
  if (final_loss) *final_loss = last / ((double)batch * M->n_in);
  return AX_OK;
}

int ax_mlp_gather_pairs(const ax_mlp *M, const double *r, const double *err, const double *minv,
                        const int *idx, int nsamples, float *X, float *T, void *stream) {
  if (!M || !r || !err || !minv || !idx || nsamples < 0 || !X || !T) return AX_EINVAL;
  if (nsamples == 0) return AX_OK;
  gather_pairs_kernel<<<nsamples, kThreads, 0, (cudaStream_t)stream>>>(X, T, r, err, minv, idx,
                                                                       M->n_in);
  return ax::launch_status();
}

}  // extern "C"
