// Fused z pass of one relaxation iteration for FP32 mesh data (Secs. III.B-C).
// This file holds the arithmetic and the host side; the kernel is k_relax_rows (relax_rows.cuh).
//
// A CTA owns TY = 16 consecutive rows (x, y0 .. y0 + 15) of the mesh.  It
//   1. inverse-transforms along z the six y-inverted spectra of those rows as
//      three field pairs (two real fields per complex pencil), in the order
//        A = (H_xy, H_xz),  B = (H_yz, N),  C = (a, b), two of H_xx, H_yy, H_zz,
//      and folds them into one accumulator per point,
//        after A and B:  r = -2 (H_xy^2 + H_xz^2 + H_yz^2) + c2 N,
//      then with the mean-free d = D - <D>, u = a + b and the third diagonal one, d - u (the trace
//      identity):
//        R  = r + 2 a b + 2 u (d - u) + alpha d - S         (Eq. FullDGP2, LHS - RHS)
//      (-2 sum_{i<j} (H_ij^2 - H_ii H_jj) = -2 (H_xy^2 + H_xz^2 + H_yz^2) + 2 a b + 2 u (d - u));
//        B' = d ((1 - w) d + alpha) - R                     (Eq. Bwpara)
//        Delta = (alpha + 2 (1 - w) d)^2 - 4 (1 - w) R      (= alpha^2 + 4 (1 - w) B')
//      bad points (Delta < 0) take Delta = 0 (Sec. III.C), and
//        D_new = 2 B' / (alpha + sqrt(Delta))              (Eq. nabla^2Cwpara, '+' root);
//   2. writes D_new and forward-transforms it along z into the transposed half
//      spectrum, ready for the next iteration's y pass;
//   3. emits FP64 block partials of sum |R|, sum D_new, bad points, non-finite R.
// The arithmetic of r, R, B' and Delta is a policy: FP32; FP32 with an exact
// discriminant and pair sums (the mixed default); pairs of floats with
// error-free transformations for R and Delta (about 48 significant bits); or FP64.
//
// Data movement.  The spectra are read as TMA tiles (one tensor map per
// spectrum; a tile is 16 complex values along y, 128 bytes, for every kz),
// landed with the 128-byte swizzle so that the transform's column reads are
// free of bank conflicts, and completed on an mbarrier.  Two tile buffers
// alternate: while one pair is transformed the next lands in the other; the
// four-step transpose of a pair reuses the bytes of the tile it came from.
// The rows of D and S come in by plain bulk copies into padded rows.  Every
// wait is bounded (tma.cuh): on expiry the CTA records a fault that stops the
// solve with DGP_E_TIMEOUT, waits for the copies it issued and returns.
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <cudaTypedefs.h>

#include <mutex>
#include <type_traits>

#include "eft.cuh"
#include "fft_core.cuh"
#include "kernels.cuh"
#include "tma.cuh"

namespace dgp {

// ---------------------------------------------------------------- arithmetic policies
__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float fdiv_full(float a, float b) {
  float r;
  asm("div.full.ftz.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

struct PointOut {
  float bp, dt;  // B' and Delta, rounded to float
  bool neg;      // Delta < 0 (a bad point)
};

struct RxF32 {
  using Acc = float;
  using Sum = float;
  static constexpr bool kApproxRoot = true;
  __device__ static void pair_a(Acc& r, float x, float y) { r = fmaf(-2.f * x, x, (-2.f * y) * y); }
  __device__ static void pair_b(Acc& r, float x, float n, const RelaxParams& rp) {
    r = fmaf(-2.f * x, x, fmaf(rp.c2_hi, n, r));
  }
  __device__ static PointOut finish(Acc r, float a, float b, float D, float S, float m_hi, float, double,
                                    const RelaxParams& rp, Sum& rsum, float& nonfin) {
    const float d = D - m_hi, u = a + b, c = d - u;
    const float R = fmaf(2.f * a, b, fmaf(2.f * u, c, fmaf(rp.alpha_hi, d, r - S)));
    PointOut o;
    o.bp = fmaf(d, fmaf(rp.omw, d, rp.alpha_hi), -R);
    const float s = fmaf(rp.two_omw, d, rp.alpha_hi);
    o.dt = fmaf(s, s, -rp.four_omw_hi * R);
    o.neg = o.dt < 0.f;
    if (isfinite(R)) rsum += fabsf(R);
    else nonfin += 1.f;
    return o;
  }
};

// Config-3 mixed arithmetic: R, B' and D_new in FP32 (the FP32 data's own
// rounding already leaves a residual floor of order 1e-8 of <|S|>, which
// pair arithmetic cannot go below); the discriminant's sign from Delta formed
// exactly for the FP32 s = alpha + 2 (1 - w) d and R (a pair); the per-thread
// sum of D_new (its mean is removed next iteration) as a pair; every
// cross-thread sum in FP64.
struct RxM32 {
  using Acc = float;
  using Sum = float;
  static constexpr bool kApproxRoot = true;
  __device__ static void pair_a(Acc& r, float x, float y) { RxF32::pair_a(r, x, y); }
  __device__ static void pair_b(Acc& r, float x, float n, const RelaxParams& rp) { RxF32::pair_b(r, x, n, rp); }
  __device__ static PointOut finish(Acc r, float a, float b, float D, float S, float m_hi, float, double,
                                    const RelaxParams& rp, Sum& rsum, float& nonfin) {
    const float d = D - m_hi, u = a + b, c = d - u;
    const float R = fmaf(2.f * a, b, fmaf(2.f * u, c, fmaf(rp.alpha_hi, d, r - S)));
    PointOut o;
    o.bp = fmaf(d, fmaf(rp.omw, d, rp.alpha_hi), -R);
    const float s = fmaf(rp.two_omw, d, rp.alpha_hi);
    FP v = fp_prod(s, s);
    FP t = fp_prod(-rp.four_omw_hi, R);
    t.lo = fmaf(-rp.four_omw_lo, R, t.lo);
    fp_acc(v, t);
    v = fp_fast(v.hi, v.lo);
    o.neg = v.hi < 0.f || (v.hi == 0.f && v.lo < 0.f);
    o.dt = v.hi + v.lo;
    if (isfinite(R)) rsum += fabsf(R);
    else nonfin += 1.f;
    return o;
  }
};

struct RxEFT {
  using Acc = FP;
  using Sum = FP;
  static constexpr bool kApproxRoot = false;
  __device__ static void pair_a(Acc& r, float x, float y) {
    r = fp_prod(-2.f * x, x);
    fp_acc(r, fp_prod(-2.f * y, y));
  }
  __device__ static void pair_b(Acc& r, float x, float n, const RelaxParams& rp) {
    fp_acc(r, fp_prod(-2.f * x, x));
    FP c = fp_prod(rp.c2_hi, n);
    c.lo = fmaf(rp.c2_lo, n, c.lo);
    fp_acc(r, c);
  }
  __device__ static PointOut finish(Acc r, float a, float b, float D, float S, float m_hi, float m_lo, double,
                                    const RelaxParams& rp, Sum& rsum, float& nonfin) {
    FP d = fp_two_sum(D, -m_hi);
    d.lo -= m_lo;
    d = fp_fast(d.hi, d.lo);
    const FP u = fp_two_sum(a, b);  // a + b exactly
    FP c = fp_two_sum(d.hi, -u.hi);  // the third diagonal one, d - u
    c.lo += d.lo - u.lo;
    fp_acc(r, fp_prod(2.f * a, b));
    {
      FP p = fp_prod(2.f * u.hi, c.hi);
      p.lo = fmaf(2.f * u.hi, c.lo, fmaf(2.f * u.lo, c.hi, p.lo));
      fp_acc(r, p);
    }
    {
      FP p = fp_prod(rp.alpha_hi, d.hi);
      p.lo = fmaf(rp.alpha_hi, d.lo, fmaf(rp.alpha_lo, d.hi, p.lo));
      fp_acc(r, p);
    }
    fp_acc(r, FP{-S, 0.f});
    const FP R = fp_fast(r.hi, r.lo);
    PointOut o;
    // B' only feeds D_new, an FP32 datum: FP32 from the pair-accurate R and d suffices
    o.bp = fmaf(d.hi, fmaf(rp.omw, d.hi, rp.alpha_hi), -R.hi);
    {
      const float s = fmaf(rp.two_omw, d.hi, rp.alpha_hi);
      FP v = fp_prod(s, s);
      FP t = fp_prod(-rp.four_omw_hi, R.hi);
      t.lo = fmaf(-rp.four_omw_hi, R.lo, fmaf(-rp.four_omw_lo, R.hi, t.lo));
      fp_acc(v, t);
      v = fp_fast(v.hi, v.lo);
      o.neg = v.hi < 0.f || (v.hi == 0.f && v.lo < 0.f);
      o.dt = v.hi + v.lo;
    }
    if (isfinite(R.hi)) fp_acc(rsum, R.hi < 0.f ? FP{-R.hi, -R.lo} : R);
    else nonfin += 1.f;
    return o;
  }
};

// Bound by the FP64 pipe, so r carries half of the sum (factors of two are folded into one FMA at the
// end): 17 FP64 operations a point instead of 28.
struct RxF64 {
  using Acc = double;
  using Sum = double;
  static constexpr bool kApproxRoot = false;
  __device__ static void pair_a(Acc& r, float x, float y) {
    const double u = (double)x, v = (double)y;
    r = fma(u, u, v * v);
  }
  __device__ static void pair_b(Acc& r, float x, float n, const RelaxParams& rp) {
    const double u = (double)x;
    r = fma(-u, u, fma(0.5 * rp.c2, (double)n, -r));
  }
  __device__ static PointOut finish(Acc r, float fa, float fb, float D, float S, float, float, double mean,
                                    const RelaxParams& rp, Sum& rsum, float& nonfin) {
    const double a = (double)fa, b = (double)fb;
    const double d = (double)D - mean, u = a + b, c = d - u;
    const double h = fma(a, b, fma(u, c, r));
    const double R = fma(2.0, h, fma(rp.alpha, d, -(double)S));
    const double omw = 1.0 - rp.w;
    PointOut o;
    o.bp = (float)fma(d, fma(omw, d, rp.alpha), -R);
    const double s = fma(2.0 * omw, d, rp.alpha);
    const double v = fma(s, s, (-4.0 * omw) * R);
    o.neg = v < 0.0;
    o.dt = (float)v;
    if (isfinite(R)) rsum += fabs(R);
    else nonfin += 1.f;
    return o;
  }
};

}  // namespace dgp

#include "relax_rows.cuh"

namespace dgp {

// ---------------------------------------------------------------- host side
static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    else
      cudaGetLastError();
  });
  return fn;
}

template <int N>
int relax_maps(float2* const* spec6, float2* const* snew2, RelaxMaps* out) {
  using G = RowGeom<N, false>;  // boxes and tiles are the same for wide rows
  const PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
  if (!enc) return 1;
  // the half spectrum S[kz][x][y] as floats: dim 0 = 2N floats along y, dim 1 = x, dim 2 = kz
  const cuuint64_t dims[3] = {(cuuint64_t)2 * N, (cuuint64_t)N, (cuuint64_t)G::NK};
  const cuuint64_t strides[2] = {(cuuint64_t)2 * N * 4, (cuuint64_t)N * 2 * N * 4};
  const cuuint32_t box[3] = {(cuuint32_t)2 * G::TY, 1, (cuuint32_t)G::BOXK};
  const cuuint32_t es[3] = {1, 1, 1};
  out->out[0] = snew2[0];
  out->out[1] = snew2[1];
  for (int f = 0; f < 8; ++f) {
    const CUresult r = enc(f < 6 ? &out->map[f] : &out->out_map[f - 6], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3,
                           f < 6 ? spec6[f] : snew2[f - 6], dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return 1;
  }
  return 0;
}

void relax_set_maps(const RelaxMaps& maps, float2* Snew, RelaxTmaArgs* a) {
  memcpy(a->map, maps.map, sizeof(a->map));
  a->out_map = maps.out_map[Snew == maps.out[0] ? 0 : 1];
}

template <int N> int relax_tma_blocks() { return (N / RowGeom<N, false>::TY) * N; }

template <int N, class AR, int RB>
static void launch_rt(const RelaxTmaArgs* a, int count, const float2* tw, cudaStream_t s) {
  RelaxTmaBatch<RB> b;
  for (int r = 0; r < count; ++r) b.a[r] = a[r];
  using W = RowWide<N, AR, RB>;
  using G = typename W::G;
  raise_smem_limit<k_relax_rows<N, AR, RB>>(W::SMEM);
  k_relax_rows<N, AR, RB><<<dim3(N / G::TY, N, count), G::THREADS, W::SMEM, s>>>(b, tw);
}

template <int N, class AR>
static void launch_rt(const RelaxTmaArgs* a, int count, bool of_class, const float2* tw, cudaStream_t s) {
  if (of_class) launch_rt<N, AR, kBatchMax>(a, count, tw, s);
  else launch_rt<N, AR, 1>(a, 1, tw, s);
}

template <int N>
void launch_relax_tma(int arith, const RelaxMaps& maps, const float* D, const double* dsum, const float* S,
                      float* Dnew, float2* Snew, RelaxParams rp, double* partials, const float2* tw, cudaStream_t s,
                      const int* skip, int* fault, unsigned long long wait_ns, int withhold) {
  RelaxTmaArgs a;
  relax_set_maps(maps, Snew, &a);
  a.D = D; a.dsum = dsum; a.S = S; a.Dnew = Dnew; a.partials = partials; a.rp = rp;
  a.skip = skip; a.fault = fault; a.wait_ns = wait_ns; a.withhold = withhold;
  launch_relax_tma_batch<N>(arith, &a, 1, false, tw, s);
}

template <int N>
void launch_relax_tma_batch(int arith, const RelaxTmaArgs* a, int count, bool of_class, const float2* tw,
                            cudaStream_t s) {
  if (count < 1 || count > (of_class ? kBatchMax : 1)) return;
  if (arith == ARITH_F64) launch_rt<N, RxF64>(a, count, of_class, tw, s);
  else if (arith == ARITH_EFT) launch_rt<N, RxEFT>(a, count, of_class, tw, s);
  else if (arith == ARITH_M32) launch_rt<N, RxM32>(a, count, of_class, tw, s);
  else launch_rt<N, RxF32>(a, count, of_class, tw, s);
}

#define DGP_INST_RT(N)                                                                                          \
  template int relax_maps<N>(float2* const*, float2* const*, RelaxMaps*);                                     \
  template int relax_tma_blocks<N>();                                                                         \
  template void launch_relax_tma<N>(int, const RelaxMaps&, const float*, const double*, const float*, float*,  \
                                    float2*, RelaxParams, double*, const float2*, cudaStream_t, const int*, int*, \
                                    unsigned long long, int);                                                 \
  template void launch_relax_tma_batch<N>(int, const RelaxTmaArgs*, int, bool, const float2*, cudaStream_t);
DGP_INST_RT(16)
DGP_INST_RT(32)
DGP_INST_RT(48)
DGP_INST_RT(64)
DGP_INST_RT(96)
DGP_INST_RT(128)
DGP_INST_RT(256)
DGP_INST_RT(512)

}  // namespace dgp
