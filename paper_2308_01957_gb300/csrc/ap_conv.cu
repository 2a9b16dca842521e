// Direct PSF correlation through shared memory, with the model / residual /
// chi^2 epilogue (forward) or a plain store (adjoint), and the deterministic
// float64 gathers of chi^2 and gradient partials.
//
// Paper: Sec. "PSF convolution" (direct mode, PSF normalised before
// convolution), Eq. chi2 and the variance / mask maps of Sec. "chi^2
// Optimization".
//
// Both directions are the same correlation
//     out(y, x) = sum_{ty < K, tx < K} Pk[ty][tx] * in(y + ty + off, x + tx + off)
// with in() zero outside its array:
//   forward: in = galaxy layer G (image grown by h), Pk = flipped PSF, off = 0,
//            which is the true convolution M = P * G on the image pixels;
//   adjoint: in = w r on the image, Pk = PSF, off = -2h, out = the galaxy
//            layer; the transpose of the forward map.
//
// Thread layout: a thread owns RY rows x RX = 4 columns of outputs.  For
// every input row it slides a register window of 8 values along the row in
// steps of 4 (one 16-byte shared load per step) and reads the matching PSF
// row chunk for each of its output rows as a broadcast 16-byte load, so the
// loop issues 16 RY FMAs per RY + 1 shared-memory loads.  Tile variants
// (threads BX x BY, RY) are picked per problem by timing them (autotuner in
// ap_api.cu).
#include <vector>

#include "ap_internal.cuh"

namespace ap {

constexpr int RX = 4;

template <typename T> struct Limits;
template <> struct Limits<float> { __device__ static constexpr float max_finite() { return 3.402823466e38f; } };
template <> struct Limits<double> { __device__ static constexpr double max_finite() { return 1.7976931348623157e308; } };

template <typename T> struct Vec4;
template <> struct Vec4<float> {
  __device__ __forceinline__ static void ld(const float* p, float& a, float& b, float& c, float& d) {
    float4 v = *reinterpret_cast<const float4*>(p);
    a = v.x; b = v.y; c = v.z; d = v.w;
  }
};
template <> struct Vec4<double> {
  __device__ __forceinline__ static void ld(const double* p, double& a, double& b, double& c, double& d) {
    double2 v0 = *reinterpret_cast<const double2*>(p);
    double2 v1 = *reinterpret_cast<const double2*>(p + 2);
    a = v0.x; b = v0.y; c = v1.x; d = v1.y;
  }
};

// variant table: threads BX x BY, rows per thread RY
struct ConvShape { int bx, by, ry; };
// (the first one for small images: a 128^2 image makes 64 CTAs of it, 16 of the
// next larger one)
static const ConvShape kShapes[N_CONV_VARIANTS] = {{8, 8, 1}, {16, 8, 4}, {8, 16, 4}, {16, 16, 2}, {16, 8, 8}, {32, 8, 4},
                                                   {16, 8, 2}};
int conv_tile_w(int v) { return kShapes[v].bx * RX; }
int conv_tile_h(int v) { return kShapes[v].by * kShapes[v].ry; }
int conv_threads(int v) { return kShapes[v].bx * kShapes[v].by; }

// The tile's input window and PSF into shared memory by asynchronous copies, all
// in flight together (through registers every round of the loop waited for its
// load: 13 of the 17 us of a 128^2 image's correlation).  Outside the input the
// copies fill zeros.
template <typename T>
__device__ __forceinline__ void copy_async(unsigned dst, const T* src, bool in) {
  if constexpr (sizeof(T) == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(in ? 4 : 0) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(in ? 8 : 0) : "memory");
}
template <typename T, int NT>
__device__ __forceinline__ void load_tile(const T* __restrict__ in, int Hi, int Wi, int in_r0, int in_c0,
                                          const T* __restrict__ pk, int n_pk, T* s_in, T* s_pk, int SH, int SW) {
  const int tid = threadIdx.x;
  const unsigned d_pk = (unsigned)__cvta_generic_to_shared(s_pk), d_in = (unsigned)__cvta_generic_to_shared(s_in);
  constexpr int V = 16 / sizeof(T);   // PSF rows are whole 16-byte words
#pragma unroll 2
  for (int idx = tid * V; idx < n_pk; idx += NT * V)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d_pk + idx * (unsigned)sizeof(T)), "l"(pk + idx)
                 : "memory");
#pragma unroll 4
  for (int idx = tid; idx < SH * SW; idx += NT) {
    const int r = idx / SW, c = idx - r * SW;
    const int gr = in_r0 + r, gc = in_c0 + c;
    const bool inside = gr >= 0 && gr < Hi && gc >= 0 && gc < Wi;
    copy_async<T>(d_in + idx * (unsigned)sizeof(T), in + (inside ? (size_t)gr * Wi + gc : 0), inside);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
}

template <typename T, int BX, int BY, int RY>
__device__ __forceinline__ void corr_tile(const T* __restrict__ in, int Hi, int Wi, int in_r0, int in_c0,
                                          const T* __restrict__ pk, int K, int K4, T* smem,
                                          T (&acc)[RY][RX]) {
  constexpr int NT = BX * BY;
  constexpr int TW = BX * RX, TH = BY * RY;
  const int SW = TW + K4;           // shared row stride (multiple of 4)
  const int SH = TH + K - 1;
  T* s_in = smem;
  T* s_pk = smem + SH * SW;
  const int tid = threadIdx.x;
  load_tile<T, NT>(in, Hi, Wi, in_r0, in_c0, pk, K * K4, s_in, s_pk, SH, SW);
  const int lx = tid % BX, ly = tid / BX;
#pragma unroll
  for (int a = 0; a < RY; ++a)
#pragma unroll
    for (int b = 0; b < RX; ++b) acc[a][b] = (T)0;
  const int nchunk = K4 >> 2;
  for (int ir = 0; ir < RY + K - 1; ++ir) {
    const T* row = s_in + (ly * RY + ir) * SW + lx * RX;
    T w0, w1, w2, w3, w4, w5, w6, w7;
    Vec4<T>::ld(row, w0, w1, w2, w3);
    for (int c = 0; c < nchunk; ++c) {
      Vec4<T>::ld(row + 4 * c + 4, w4, w5, w6, w7);
#pragma unroll
      for (int ry = 0; ry < RY; ++ry) {
        const int ty = ir - ry;
        if (ty >= 0 && ty < K) {
          T p0, p1, p2, p3;
          Vec4<T>::ld(s_pk + ty * K4 + 4 * c, p0, p1, p2, p3);
          acc[ry][0] = fma(p3, w3, fma(p2, w2, fma(p1, w1, fma(p0, w0, acc[ry][0]))));
          acc[ry][1] = fma(p3, w4, fma(p2, w3, fma(p1, w2, fma(p0, w1, acc[ry][1]))));
          acc[ry][2] = fma(p3, w5, fma(p2, w4, fma(p1, w3, fma(p0, w2, acc[ry][2]))));
          acc[ry][3] = fma(p3, w6, fma(p2, w5, fma(p1, w4, fma(p0, w3, acc[ry][3]))));
        }
      }
      w0 = w4; w1 = w5; w2 = w6; w3 = w7;
    }
  }
}

// two float32 products and additions in one instruction (the same roundings as
// two fmaf)
__device__ __forceinline__ void fma2(float2& acc, float2 a, float2 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;"
      : "+l"(reinterpret_cast<unsigned long long&>(acc))
      : "l"(reinterpret_cast<const unsigned long long&>(a)), "l"(reinterpret_cast<const unsigned long long&>(b)));
}

// Fast path for float and PSF rows of NC = K4/4 chunks known at compile time:
// the whole input-row window of 4 NC + 4 values is loaded once per input row
// (NC + 1 shared loads).  Two output rows y, y + 1 share an input row with the PSF
// rows ty and ty - 1, so their products are packed: the PSF is kept as pairs
// (P[ty], P[ty - 1]), the window's values are duplicated in registers, and every
// tap chunk of a row pair is an unrolled block of 16 two-way FMAs -- the loop was
// bound by instruction issue (3.1 to 3.4 of 4 per clock, the FMA pipe 63 to 70 %
// busy), and this issues half the FMAs.  The first and the last input row of a pair
// belong to one of its rows only and take plain FMAs (a zero weight would carry an
// infinite input into the other row).  The order of the additions is that of the
// plain loop.  Four 1024^2 exposures, 31 px PSFs: forward 180 -> 167 us, adjoint
// 171 -> 161 us; twelve of 2048^2: 1370 -> 1270 and 1790 -> 1690.
template <int BX, int BY, int RY, int NC>
__device__ __forceinline__ void corr_tile_nc(const float* __restrict__ in, int Hi, int Wi, int in_r0, int in_c0,
                                             const float* __restrict__ pk, int K, float* smem,
                                             float (&acc)[RY][RX]) {
  constexpr int NT = BX * BY;
  constexpr int TW = BX * RX, TH = BY * RY;
  constexpr int K4 = 4 * NC;
  constexpr int SW = TW + K4;
  static_assert(RY % 2 == 0, "rows in pairs");
  const int SH = TH + K - 1;
  float* s_in = smem;
  float* s_pk = smem + SH * SW;                                  // pairs (P[ty], P[ty - 1]), ty = 0 .. K
  const int tid = threadIdx.x;
  for (int idx = tid; idx < (K + 1) * K4; idx += NT) {
    const int ty = idx / K4;
    reinterpret_cast<float2*>(s_pk)[idx] =
        make_float2(ty < K ? __ldg(pk + idx) : 0.f, ty > 0 ? __ldg(pk + idx - K4) : 0.f);
  }
  load_tile<float, NT>(in, Hi, Wi, in_r0, in_c0, pk, 0, s_in, s_pk, SH, SW);
  const int lx = tid % BX, ly = tid / BX;
  float2 a2[RY / 2][RX];
#pragma unroll
  for (int a = 0; a < RY / 2; ++a)
#pragma unroll
    for (int b = 0; b < RX; ++b) a2[a][b] = make_float2(0.f, 0.f);
  for (int ir = 0; ir < RY + K - 1; ++ir) {
    const float* row = s_in + (ly * RY + ir) * SW + lx * RX;
    float w[4 * NC + 4];
#pragma unroll
    for (int c = 0; c <= NC; ++c) Vec4<float>::ld(row + 4 * c, w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
#pragma unroll
    for (int q = 0; q < RY / 2; ++q) {
      const int ty = ir - 2 * q;
      if (ty < 0 || ty > K) continue;
      const float* prow = s_pk + 2 * ty * K4;
      if (ty > 0 && ty < K) {
#pragma unroll
        for (int c = 0; c < 2 * NC; ++c) {   // two taps per 16-byte load
          float2 p0, p1;
          Vec4<float>::ld(prow + 4 * c, p0.x, p0.y, p1.x, p1.y);
#pragma unroll
          for (int rx = 0; rx < RX; ++rx) {
            fma2(a2[q][rx], p0, make_float2(w[2 * c + rx], w[2 * c + rx]));
            fma2(a2[q][rx], p1, make_float2(w[2 * c + rx + 1], w[2 * c + rx + 1]));
          }
        }
      } else {
        const bool up = ty == 0;   // row 2q alone; else (ty == K) row 2q + 1 alone
        float v[RX];
#pragma unroll
        for (int rx = 0; rx < RX; ++rx) v[rx] = up ? a2[q][rx].x : a2[q][rx].y;
#pragma unroll
        for (int c = 0; c < 2 * NC; ++c) {
          float2 p0, p1;
          Vec4<float>::ld(prow + 4 * c, p0.x, p0.y, p1.x, p1.y);
          const float pa = up ? p0.x : p0.y, pb = up ? p1.x : p1.y;
#pragma unroll
          for (int rx = 0; rx < RX; ++rx) v[rx] = fmaf(pb, w[2 * c + rx + 1], fmaf(pa, w[2 * c + rx], v[rx]));
        }
#pragma unroll
        for (int rx = 0; rx < RX; ++rx) {
          if (up) a2[q][rx].x = v[rx];
          else a2[q][rx].y = v[rx];
        }
      }
    }
  }
#pragma unroll
  for (int a = 0; a < RY / 2; ++a)
#pragma unroll
    for (int b = 0; b < RX; ++b) {
      acc[2 * a][b] = a2[a][b].x;
      acc[2 * a + 1][b] = a2[a][b].y;
    }
}

// dispatch between the generic (runtime K4) tile and the NC-templated one
template <typename T, int BX, int BY, int RY, int NC>
__device__ __forceinline__ void corr_any(const T* __restrict__ in, int Hi, int Wi, int in_r0, int in_c0,
                                         const T* __restrict__ pk, int K, int K4, T* smem, T (&acc)[RY][RX]) {
  if constexpr (NC > 0 && sizeof(T) == 4) {
    corr_tile_nc<BX, BY, RY, NC>(reinterpret_cast<const float*>(in), Hi, Wi, in_r0, in_c0,
                                 reinterpret_cast<const float*>(pk), K, reinterpret_cast<float*>(smem),
                                 reinterpret_cast<float(&)[RY][RX]>(acc));
  } else {
    corr_tile<T, BX, BY, RY>(in, Hi, Wi, in_r0, in_c0, pk, K, K4, smem, acc);
  }
}

// forward: model = P * G + U, r = d - m, w = mask ? 0 : 1/var, chi^2 partial,
// w r stored for the adjoint; model optionally stored
template <typename T, int BX, int BY, int RY, int NC>
__global__ void __launch_bounds__(BX * BY) forward_conv_kernel(const ConvWork* __restrict__ work,
                                                               const ImageDev* __restrict__ imgs,
                                                               double* __restrict__ chi2_partial,
                                                               const __grid_constant__ ModelOut model_out,
                                                               const int* __restrict__ skip, int trial,
                                                               int store_sw, int* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* smem = reinterpret_cast<T*>(smem_raw);
  __shared__ double red[32];
  const ConvWork w = work[blockIdx.x];
  const ImageDev& im = imgs[w.image];
  if (skip && skip[im.group]) return;   // w r already holds this point; the gather keeps its chi^2
  T acc[RY][RX];
  if (im.has_gal) {
    corr_any<T, BX, BY, RY, NC>((const T*)im.gal, im.Hp, im.Wp, w.r0, w.c0, (const T*)im.psf_flip, im.K, im.K4,
                                smem, acc);
  } else {
#pragma unroll
    for (int a = 0; a < RY; ++a)
#pragma unroll
      for (int b = 0; b < RX; ++b) acc[a][b] = (T)0;
  }
  const int lx = threadIdx.x % BX, ly = threadIdx.x / BX;
  const T* __restrict__ U = (const T*)im.unc;
  const float* __restrict__ data = im.data;
  const float* __restrict__ varp = im.var;
  const uint8_t* __restrict__ mask = im.mask;
  T* WR = (T*)(trial ? im.wr_trial : im.wr);
  float* SW = sizeof(T) == 4 && store_sw ? im.sw : nullptr;
  T* M = (T*)(model_out.n > 0 ? model_out.p[w.image] : model_out.table ? model_out.table[w.image] : nullptr);
  // per-pixel residual math in T (float64 is scarce on this GPU); the
  // thread's chi^2 partial of at most RY * 4 terms joins the block sum in
  // float64.  A row's inputs are all loaded before its first store.
  T c2t = (T)0;
  int bad = 0;
#pragma unroll
  for (int ry = 0; ry < RY; ++ry) {
    const int oi = w.r0 + ly * RY + ry;
    if (oi >= im.H) break;
    const int oj0 = w.c0 + lx * RX;
    const size_t o0 = (size_t)oi * im.W + oj0;
    T u[RX];
    float dv[RX], vv[RX];
    int mk[RX];
#pragma unroll
    for (int rx = 0; rx < RX; ++rx) {
      const bool in = oj0 + rx < im.W;
      u[rx] = in ? __ldg(U + o0 + rx) : (T)0;
      dv[rx] = in ? __ldg(data + o0 + rx) : 0.f;
      vv[rx] = in ? __ldg(varp + o0 + rx) : 1.f;
      mk[rx] = in && mask != nullptr ? (int)__ldg(mask + o0 + rx) : 0;
    }
#pragma unroll
    for (int rx = 0; rx < RX; ++rx) {
      if (oj0 + rx < im.W) {
        const size_t o = o0 + rx;
        const T m = acc[ry][rx] + u[rx];
        if (M) M[o] = m;
        const T r = (T)dv[rx] - m;
        const T var = (T)vv[rx];
        T wt = (T)0;
        if (mk[rx] == 0) {
          if (var > (T)0 && var <= Limits<T>::max_finite()) wt = (T)1 / var;
          else bad = 1;
        }
        const T wr = wt * r;
        c2t += wr * r;
        WR[o] = wr;
        // sqrt(w) for the Jacobian columns (correctly rounded division and root)
        if (SW) SW[o] = wt > (T)0 ? 1.0f / sqrtf((float)var) : 0.f;
      }
    }
  }
  double c2 = (double)c2t;
  if (bad) atomicCAS(status, 0, AP_ERR_NONFINITE);
  if (chi2_partial) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c2 += __shfl_xor_sync(0xffffffffu, c2, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) red[warp] = c2;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int k = 0; k < (BX * BY + 31) / 32; ++k) s += red[k];
      chi2_partial[blockIdx.x] = s;
    }
  }
}

// adjoint: adj(ip, jp) = sum P[ty][tx] wr(ip + ty - 2h, jp + tx - 2h) on the galaxy layer
template <typename T, int BX, int BY, int RY, int NC>
__global__ void __launch_bounds__(BX * BY) adjoint_conv_kernel(const ConvWork* __restrict__ work,
                                                               const ImageDev* __restrict__ imgs) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* smem = reinterpret_cast<T*>(smem_raw);
  const ConvWork w = work[blockIdx.x];
  const ImageDev& im = imgs[w.image];
  T acc[RY][RX];
  corr_any<T, BX, BY, RY, NC>((const T*)im.wr, im.H, im.W, w.r0 - 2 * im.h, w.c0 - 2 * im.h, (const T*)im.psf_norm,
                              im.K, im.K4, smem, acc);
  const int lx = threadIdx.x % BX, ly = threadIdx.x / BX;
  T* A = (T*)im.adj;
#pragma unroll
  for (int ry = 0; ry < RY; ++ry) {
    const int oi = w.r0 + ly * RY + ry;
    if (oi >= im.Hp) break;
#pragma unroll
    for (int rx = 0; rx < RX; ++rx) {
      const int oj = w.c0 + lx * RX + rx;
      if (oj < im.Wp) A[(size_t)oi * im.Wp + oj] = acc[ry][rx];
    }
  }
}

// Jacobian columns of convolved sources: J_k = P * (d G_s / d theta_k) on the
// source's Jacobian support (its sampling box grown by h, clipped to the
// image), from the stored derivative images.  One CTA per output tile of one
// source, looping over the source's free slots.  The float path stores
// sqrt(w) J_k into the column blocks, the float64 path J_k row by row.
template <typename T, int BX, int BY, int RY, int NC>
__global__ void __launch_bounds__(BX * BY) jcol_kernel(const JcolWork* __restrict__ work,
                                                       const SourceDev* __restrict__ srcs,
                                                       const ImageDev* __restrict__ imgs, const T* __restrict__ dbuf,
                                                       T* __restrict__ jbuf) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* smem = reinterpret_cast<T*>(smem_raw);
  const JcolWork w = work[blockIdx.x];
  const SourceDev& sd = srcs[w.src];
  const ImageDev& im = imgs[sd.image];
  const int bh = sd.box[1] - sd.box[0], bw = sd.box[3] - sd.box[2];
  const int64_t barea = (int64_t)bh * bw;
  const int sh = sd.sup[1] - sd.sup[0], sw = sd.sup[3] - sd.sup[2];
  const int64_t sarea = (int64_t)sh * sw;
  const int lx = threadIdx.x % BX, ly = threadIdx.x / BX;
  int f = 0;
  for (int k = 0; k < sd.nslot; ++k) {
    if (sd.pidx[k] < 0) continue;
    T acc[RY][RX];
    corr_any<T, BX, BY, RY, NC>(dbuf + sd.d_off + k * barea, bh, bw, w.r0 - im.h - sd.box[0],
                                w.c0 - im.h - sd.box[2], (const T*)im.psf_flip, im.K, im.K4, smem, acc);
#pragma unroll
    for (int ry = 0; ry < RY; ++ry) {
      const int oi = w.r0 + ly * RY + ry;
      if (oi >= sd.sup[1]) break;
#pragma unroll
      for (int rx = 0; rx < RX; ++rx) {
        const int oj = w.c0 + lx * RX + rx;
        if (oj >= sd.sup[3]) break;
        if constexpr (sizeof(T) == 4)
          jbuf[col_block(sd, f, oi, oj)] = acc[ry][rx] * im.sw[(size_t)oi * im.W + oj];
        else
          jbuf[sd.j_off + k * sarea + (int64_t)(oi - sd.sup[0]) * sw + (oj - sd.sup[2])] = acc[ry][rx];
      }
    }
    ++f;
    __syncthreads();   // the next slot reloads the shared tile
  }
}

// (an NC kernel meets K <= 4 NC only, and keeps the PSF as (K + 1) x K4 pairs)
template <typename T, int BX, int BY, int RY, int NC>
static size_t corr_smem_bytes(int Kmax) {
  const int K = NC > 0 && Kmax > 4 * NC ? 4 * NC : Kmax, K4 = NC > 0 ? 4 * NC : (K + 3) & ~3;
  return (size_t)((BY * RY + K - 1) * (BX * RX + K4) + (NC > 0 ? 2 * (K + 1) : K) * K4) * sizeof(T);
}

// compile-time PSF chunk counts of the fast path (K4/4); others run generic
__host__ __device__ constexpr bool nc_fast(int nc) { return (nc >= 1 && nc <= 8) || nc == 13; }
int conv_nc_of(int K4, int is_double) { return (!is_double && nc_fast(K4 / 4)) ? K4 / 4 : 0; }

template <typename T, int BX, int BY, int RY, int NC>
static int configure_one(int Kmax) {
  const int need = (int)corr_smem_bytes<T, BX, BY, RY, NC>(Kmax);
  const int a = allow_max_dynamic_smem(forward_conv_kernel<T, BX, BY, RY, NC>);
  const int b = allow_max_dynamic_smem(adjoint_conv_kernel<T, BX, BY, RY, NC>);
  const int c = allow_max_dynamic_smem(jcol_kernel<T, BX, BY, RY, NC>);
  return (a >= need && b >= need && c >= need) ? 1 : 0;
}

// NC dispatch: the fast instantiations exist for float only
#define AP_NC_SWITCH(T, nc, CALL, ...)                                            \
  if (sizeof(T) == 4) {                                                           \
    switch (nc) {                                                                 \
      case 1: CALL(1, __VA_ARGS__); break;                                        \
      case 2: CALL(2, __VA_ARGS__); break;                                        \
      case 3: CALL(3, __VA_ARGS__); break;                                        \
      case 4: CALL(4, __VA_ARGS__); break;                                        \
      case 5: CALL(5, __VA_ARGS__); break;                                        \
      case 6: CALL(6, __VA_ARGS__); break;                                        \
      case 7: CALL(7, __VA_ARGS__); break;                                        \
      case 8: CALL(8, __VA_ARGS__); break;                                        \
      case 13: CALL(13, __VA_ARGS__); break;                                      \
      default: CALL(0, __VA_ARGS__); break;                                       \
    }                                                                             \
  } else {                                                                        \
    CALL(0, __VA_ARGS__);                                                         \
  }

// only the three shapes of 16 x 8 threads get NC instantiations; the others run generic
__host__ __device__ constexpr bool fast_shape(int bx, int by, int ry) {
  return bx == 16 && by == 8 && (ry == 2 || ry == 4 || ry == 8);
}

#define AP_CONV_SWITCH(v, CALL, ...)                     \
  switch (v) {                                           \
    case 0: CALL(8, 8, 1, __VA_ARGS__); break;           \
    case 1: CALL(16, 8, 4, __VA_ARGS__); break;          \
    case 2: CALL(8, 16, 4, __VA_ARGS__); break;          \
    case 3: CALL(16, 16, 2, __VA_ARGS__); break;         \
    case 4: CALL(16, 8, 8, __VA_ARGS__); break;          \
    case 5: CALL(32, 8, 4, __VA_ARGS__); break;          \
    default: CALL(16, 8, 2, __VA_ARGS__); break;         \
  }
static_assert(N_CONV_VARIANTS == 7, "AP_CONV_SWITCH lists every entry of kShapes");

template <typename T, int BX, int BY, int RY>
static int configure_variant(int Kmax) {
  int ok = configure_one<T, BX, BY, RY, 0>(Kmax);
  if constexpr (sizeof(T) == 4 && fast_shape(BX, BY, RY)) {
    ok &= configure_one<T, BX, BY, RY, 1>(Kmax);
    ok &= configure_one<T, BX, BY, RY, 2>(Kmax);
    ok &= configure_one<T, BX, BY, RY, 3>(Kmax);
    ok &= configure_one<T, BX, BY, RY, 4>(Kmax);
    ok &= configure_one<T, BX, BY, RY, 5>(Kmax);
    ok &= configure_one<T, BX, BY, RY, 6>(Kmax);
    ok &= configure_one<T, BX, BY, RY, 7>(Kmax);
    ok &= configure_one<T, BX, BY, RY, 8>(Kmax);
    ok &= configure_one<T, BX, BY, RY, 13>(Kmax);
  }
  return ok;
}

// Set the shared-memory opt-in of every tile variant for PSFs up to Kmax
// (called once per problem, outside any stream capture).  ok[v] tells whether
// variant v fits.
template <typename T>
void configure_conv(int Kmax, int* ok) {
  const int kmax = Kmax < 1 ? 1 : Kmax;
  for (int v = 0; v < N_CONV_VARIANTS; ++v) {
    int r = 0;
#define AP_CFG(BX, BY, RY, dummy) r = configure_variant<T, BX, BY, RY>(kmax)
    AP_CONV_SWITCH(v, AP_CFG, 0)
#undef AP_CFG
    // the kernel the switch launches for v must have v's tile shape (the
    // planner cuts the work items by the table)
    int same = 0;
#define AP_SAME(BX, BY, RY, dummy) same = kShapes[v].bx == BX && kShapes[v].by == BY && kShapes[v].ry == RY
    AP_CONV_SWITCH(v, AP_SAME, 0)
#undef AP_SAME
    if (ok) ok[v] = r && same;
  }
  cudaGetLastError();
}

int conv_variant_fast(int v) {
  int r = 0;
#define AP_FS(BX, BY, RY, dummy) r = fast_shape(BX, BY, RY)
  AP_CONV_SWITCH(v, AP_FS, 0)
#undef AP_FS
  return r;
}

template <typename T, int BX, int BY, int RY, int NC>
static void fwd_launch(const ConvWork* work, int n, const ImageDev* imgs, double* chi2_partial, const ModelOut& model_out,
                       const int* skip, int trial, int store_sw, int* status, int kmax, cudaStream_t st) {
  if constexpr (NC == 0 || (sizeof(T) == 4 && fast_shape(BX, BY, RY)))
    forward_conv_kernel<T, BX, BY, RY, NC><<<n, BX * BY, corr_smem_bytes<T, BX, BY, RY, NC>(kmax), st>>>(
        work, imgs, chi2_partial, model_out, skip, trial, store_sw, status);
}
template <typename T, int BX, int BY, int RY, int NC>
static void adj_launch(const ConvWork* work, int n, const ImageDev* imgs, int kmax, cudaStream_t st) {
  if constexpr (NC == 0 || (sizeof(T) == 4 && fast_shape(BX, BY, RY)))
    adjoint_conv_kernel<T, BX, BY, RY, NC><<<n, BX * BY, corr_smem_bytes<T, BX, BY, RY, NC>(kmax), st>>>(work, imgs);
}
template <typename T, int BX, int BY, int RY, int NC>
static void jc_launch(const JcolWork* work, int n, const SourceDev* srcs, const ImageDev* imgs, const T* dbuf, T* jbuf,
                      int kmax, cudaStream_t st) {
  if constexpr (NC == 0 || (sizeof(T) == 4 && fast_shape(BX, BY, RY)))
    jcol_kernel<T, BX, BY, RY, NC><<<n, BX * BY, corr_smem_bytes<T, BX, BY, RY, NC>(kmax), st>>>(work, srcs, imgs, dbuf,
                                                                                             jbuf);
}

// Launch one kernel per range of work items sharing a PSF chunk count
// (ranges[k] = {nc, start, count}); nc = 0 runs the generic tile, and a shape
// without chunk-count instantiations takes all ranges in one launch.
static std::vector<ConvRange> launch_ranges(int v, const ConvRange* ranges, int n_ranges) {
  std::vector<ConvRange> out;
  for (int k = 0; k < n_ranges; ++k) {
    if (ranges[k].count <= 0) continue;
    if (!conv_variant_fast(v) && !out.empty()) out.back().count += ranges[k].count;   // ranges lie one after another
    else out.push_back(ConvRange{conv_variant_fast(v) ? ranges[k].nc : 0, ranges[k].start, ranges[k].count});
  }
  return out;
}

template <typename T>
void launch_forward_conv(int v, const ConvWork* work, const ConvRange* ranges, int n_ranges, const ImageDev* imgs,
                         double* chi2_partial, const ModelOut& model_out, const int* skip, int trial, int store_sw,
                         int* status, int kmax, cudaStream_t st) {
  for (const ConvRange& r : launch_ranges(v, ranges, n_ranges)) {
    const int nc = r.nc;
#define AP_FWD_NC(NC, BX, BY, RY) fwd_launch<T, BX, BY, RY, NC>(work + r.start, r.count, imgs, chi2_partial + r.start, model_out, skip, trial, store_sw, status, kmax, st)
#define AP_FWD(BX, BY, RY, dummy) AP_NC_SWITCH(T, nc, AP_FWD_NC, BX, BY, RY)
    AP_CONV_SWITCH(v, AP_FWD, 0)
#undef AP_FWD
#undef AP_FWD_NC
  }
}

template <typename T>
void launch_adjoint_conv(int v, const ConvWork* work, const ConvRange* ranges, int n_ranges, const ImageDev* imgs,
                         int kmax, cudaStream_t st) {
  for (const ConvRange& r : launch_ranges(v, ranges, n_ranges)) {
    const int nc = r.nc;
#define AP_ADJ_NC(NC, BX, BY, RY) adj_launch<T, BX, BY, RY, NC>(work + r.start, r.count, imgs, kmax, st)
#define AP_ADJ(BX, BY, RY, dummy) AP_NC_SWITCH(T, nc, AP_ADJ_NC, BX, BY, RY)
    AP_CONV_SWITCH(v, AP_ADJ, 0)
#undef AP_ADJ
#undef AP_ADJ_NC
  }
}

template <typename T>
void launch_jcol(int v, const JcolWork* work, const ConvRange* ranges, int n_ranges, const SourceDev* srcs,
                 const ImageDev* imgs, const T* dbuf, T* jbuf, int kmax, cudaStream_t st) {
  for (const ConvRange& r : launch_ranges(v, ranges, n_ranges)) {
    const int nc = r.nc;
#define AP_JC_NC(NC, BX, BY, RY) jc_launch<T, BX, BY, RY, NC>(work + r.start, r.count, srcs, imgs, dbuf, jbuf, kmax, st)
#define AP_JC(BX, BY, RY, dummy) AP_NC_SWITCH(T, nc, AP_JC_NC, BX, BY, RY)
    AP_CONV_SWITCH(v, AP_JC, 0)
#undef AP_JC
#undef AP_JC_NC
  }
}

// ---------------------------------------------------------------------------
// deterministic float64 gathers: one CTA per output (its list may be long: a
// group's correlation tiles, a sky parameter's render tiles), the threads stride
// over the list in a fixed order, then a fixed tree
// ---------------------------------------------------------------------------
template <int NT, class I>
__device__ __forceinline__ double gather_sum(const double* __restrict__ partial, const I* __restrict__ idx, I k0, I k1,
                                             double* red) {
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  for (I k = k0 + threadIdx.x; k < k1; k += 4 * NT) {   // four independent gathers in flight
    I at[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) at[u] = k + u * NT < k1 ? idx[k + u * NT] : (I)-1;
#pragma unroll
    for (int u = 0; u < 4; ++u) s[u] += at[u] >= 0 ? partial[at[u]] : 0.0;
  }
  double v = (s[0] + s[1]) + (s[2] + s[3]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  v = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < NT / 32; ++w) v += red[w];
  return v;   // thread 0
}

// chi^2 of the groups (the first n_groups CTAs: scale 1; a group whose forward did
// not run keeps its value) and the gradient's components (scale -2; half the
// negative of it is J^T W r), either part may be empty: one launch for both.
constexpr int GATHER_THREADS = 128;
__global__ void __launch_bounds__(GATHER_THREADS) gather_kernel(GatherPlan g) {
  __shared__ double red[GATHER_THREADS / 32];
  const int b = blockIdx.x;
  if (b < g.n_groups) {
    if (g.skip && g.skip[b]) {
      if (threadIdx.x == 0) g.chi2[b] = g.keep[b];
      return;
    }
    const double s = gather_sum<GATHER_THREADS, int>(g.chi2_partial, g.grp_idx, g.grp_ptr[b], g.grp_ptr[b + 1], red);
    if (threadIdx.x == 0) g.chi2[b] = s;
    return;
  }
  const int p = b - g.n_groups;
  const double s =
      gather_sum<GATHER_THREADS, int64_t>(g.grad_partial, g.par_idx, g.par_ptr[p], g.par_ptr[p + 1], red);
  if (threadIdx.x == 0) {
    g.grad[p] = -2.0 * s;
    if (g.jtwr) g.jtwr[p] = s;
  }
}

void launch_gather(const GatherPlan& g, cudaStream_t st) {
  if (g.n_groups + g.n_params > 0) gather_kernel<<<g.n_groups + g.n_params, GATHER_THREADS, 0, st>>>(g);
}

template void configure_conv<float>(int, int*);
template void configure_conv<double>(int, int*);
template void launch_jcol<float>(int, const JcolWork*, const ConvRange*, int, const SourceDev*, const ImageDev*, const float*, float*, int, cudaStream_t);
template void launch_jcol<double>(int, const JcolWork*, const ConvRange*, int, const SourceDev*, const ImageDev*, const double*, double*, int, cudaStream_t);
template void launch_forward_conv<float>(int, const ConvWork*, const ConvRange*, int, const ImageDev*, double*, const ModelOut&, const int*, int, int, int*, int, cudaStream_t);
template void launch_forward_conv<double>(int, const ConvWork*, const ConvRange*, int, const ImageDev*, double*, const ModelOut&, const int*, int, int, int*, int, cudaStream_t);
template void launch_adjoint_conv<float>(int, const ConvWork*, const ConvRange*, int, const ImageDev*, int, cudaStream_t);
template void launch_adjoint_conv<double>(int, const ConvWork*, const ConvRange*, int, const ImageDev*, int, cudaStream_t);

}  // namespace ap
