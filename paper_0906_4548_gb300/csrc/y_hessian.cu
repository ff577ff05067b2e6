// Second half of the Hessian passes: from the three x-inverted spectra the Hessian x pass leaves
// (fft_x.cu), the six inputs of the relaxation, transformed back along y.
//
// Only the x component of a second derivative has to be multiplied in before the x inverse; the
// y and z components are still wavenumbers here.  With P = D(k) / k^2 the x pass therefore writes
//   G0 = IFFT_x[P],  G1 = IFFT_x[k_x P],  N = IFFT_x[-D / kbar],
// and this pass forms along each row (kz, x), k_y running over the row,
//   H_yy = k_y^2 G0,  H_zz = k_z^2 G0,  H_yz = k_y k_z G0,  H_xy = k_y G1,  H_xz = k_z G1,  N
// (Sec. III.B: nabla_ij C(k) = -k_i k_j C(k)); H_xx is D - H_yy - H_zz, the trace, in the relaxation.
// Off-diagonal pairs take |k_i k_j| when a component is on its Nyquist index.  Where that makes the
// sign depend on more than one axis, the x pass leaves small auxiliary arrays (HessAux): the
// k_x = N/2 coefficients (k_x P there counts as +N/2 in G1; H_xy needs the sign of k_y, so rows
// with k_y < 0 subtract twice that term), and IFFT_x[|k_x| P] on the column k_y = N/2 (for H_xy)
// and on the plane k_z = N/2 (for H_xz).
//
// Memory: reads three half spectra and writes six, in place: G0, G1 and N arrive in the buffers of
// H_yz, H_xz and N, each the last output formed from it, and a CTA reads only the rows it writes.
// Bound by memory: 9 half spectra (608 MB at 256^3) in 93.5 us, 0.96 of the copy rate (part of what it
// reads comes from L2).  The passes it
// replaces (an x pass writing all six spectra, then six inverse y transforms in place) moved 19 half
// spectra in 95 + 110 us; this one and the x pass move 13 in 93.5 + 67.5 us.
#include "fft_core.cuh"
#include "kernels.cuh"

namespace dgp {

template <typename T, int N> struct YHGeom {
  static constexpr int N1 = Split<N>::N1, N2 = Split<N>::N2;
  // rows per CTA, all of one kz plane.  FP32 at 256^3 with 16, 8, 4 rows and 24 warps of 80 registers
  // per SM: 131, 119, 117 us; 16 warps of 128 registers: 116, 98, 99 us.  The extra registers let a
  // thread's 16 loads and its transform overlap, which hides the latency better than more warps.
  // 512^3: 4 rows and five CTAs per SM (8 rows, two CTAs: 1061 us; 4 rows, four, five, six: 937, 898, 939).
  // FP64 at 32^3 and 48^3: 8 rows, since 4 leave half and more of a warp's lanes idle in stage one
  // (4 x 4 and 4 x 3 tasks; a 32^3 solve 2973 -> 2874 us, 48^3 7832 -> 7297).
  static constexpr int P = (sizeof(T) == 4 ? N < 512 : N == 32 || N == 48) ? 8 : 4;
  static constexpr int THREADS = P * N1;
  // row stride of the transpose (complex), N2 mod 16 when N2 < N1 so that the packed first stage's
  // rows of a half-warp fall on different banks
  static constexpr int RS0 = N1 * (N2 + 1);
  static constexpr int RS = N2 < N1 ? RS0 + ((N2 - RS0 % 16) % 16 + 16) % 16 : RS0;
  // keep the row of G0 (G1) in registers for the outputs formed from it; a 32-point first stage has
  // no room for that and reads the row again
  static constexpr bool KEEP = N <= 256;
  // CTAs of one realisation.  Below two CTAs per SM the chain of six transforms in a CTA is what takes
  // the time, so each output has threads of its own, three outputs in a CTA: those of G0 (whose buffer
  // the third overwrites), and those of G1 with N.  FP64 solves against one CTA for all outputs of a
  // field: 16^3 1750 -> 1592 us, 32^3 3221 -> 2973; FP32 the same within 1 %.  (At 96^3, four CTAs
  // per SM, splitting by the field read was slower, 14.0 against 13.2 us.)
  static constexpr int CTAS = (N / 2 + 1) * (N / P);
  static constexpr bool SPLIT = CTAS <= 304;
  static constexpr int OUTS = SPLIT ? 3 : 1;
  static constexpr size_t SMEM = sizeof(vec2_t<T>) * (N + (SPLIT ? 3 : 2) * (size_t)P * RS);
  // FP64 at 48^3, 384 threads: registers for two CTAs, since one CTA with the whole register file shuts out
  // the contexts that run beside it (six of them stepping: 12.45 -> 11.65 ms, with the passes before the
  // split 11.95; one alone: 3.37 -> 3.27 ms)
  static constexpr int MINB = sizeof(T) == 8 ? (SPLIT ? 2 : 1) : N == 512 ? 5 : SPLIT ? 1 : 512 / THREADS;
  static_assert(N % P == 0, "a CTA's rows share kz");
};

template <typename T, int RB> struct YHBatch {
  YHessArgs<T> a[RB];
};

template <typename T, int N, int RB>
__global__ void __launch_bounds__(YHGeom<T, N>::THREADS * YHGeom<T, N>::OUTS, YHGeom<T, N>::MINB)
    k_y_hessian(const __grid_constant__ YHBatch<T, RB> yb, const vec2_t<T>* __restrict__ g_tw) {
  const YHessArgs<T>& args = yb.a[RB > 1 ? blockIdx.z : 0];
  if (args.skip && *args.skip) return;
  using V = vec2_t<T>;
  using G = YHGeom<T, N>;
  constexpr int N1 = G::N1, N2 = G::N2, P = G::P;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* s_tw = reinterpret_cast<V*>(smem_raw);  // the phase table
  V* s_T = s_tw + N;                         // two transposes, alternating (SPLIT: one per output)
  for (int i = threadIdx.y * G::THREADS + threadIdx.x; i < N; i += G::THREADS * G::OUTS) s_tw[i] = g_tw[N + i];
  const int lane = threadIdx.x % N1, row = threadIdx.x / N1;
  constexpr int BPP = N / P;  // CTAs per kz plane
  // planes from the last to the first: those the x pass wrote last are still in L2 (256^3: 98 -> 93.5 us)
  const int blk = gridDim.x - 1 - blockIdx.x;
  const int kz = blk / BPP, x0 = (blk % BPP) * P;
  const int64_t plane = (int64_t)kz * N * N;
  // stage one: P x N2 tasks (a row and its column c1) on the first threads
  const int r1 = threadIdx.x / N2, c1 = threadIdx.x % N2;
  const bool act1 = N2 == N1 || threadIdx.x < P * N2;
  const int64_t row1 = plane + (int64_t)(x0 + r1) * N;
  const bool nyq_z = kz == N / 2;
  const float fz = nyq_z ? (float)(-(N / 2)) : (float)kz, fc1 = (float)c1;
  const float par = (x0 + r1) & 1 ? 2.f : -2.f;  // -2 (-1)^x
  const V* aux_x = args.aux + HessAux<N>::kx_nyq + (int64_t)kz * N;         // [ky]
  const V* aux_y = args.aux + HessAux<N>::ky_nyq + (int64_t)kz * N;         // [x]
  const V* aux_z = args.aux + HessAux<N>::kz_nyq + (int64_t)(x0 + r1) * N;  // [ky]
  V g[N1];
  __syncthreads();
  // outputs in the order H_yy, H_zz, H_yz (of G0), H_xy, H_xz (of G1), N
  const int o0 = G::SPLIT ? 3 * blockIdx.y + threadIdx.y : 0;
  const int o1 = G::SPLIT ? o0 + 1 : 6;
#pragma unroll 1
  for (int o = o0; o < o1; ++o) {
    const int slot = o == 0 ? 0 : o == 1 ? 1 : o == 2 ? 4 : o == 3 ? 2 : o == 4 ? 3 : 5;
    V* T1 = s_T + (G::SPLIT ? threadIdx.y : o & 1) * (P * G::RS);
    if (act1) {
      if (!G::KEEP || G::SPLIT || o == 0 || o == 3 || o == 5 || (o == 4 && nyq_z)) {
        const V* src = o < 3 ? args.f[4] + row1 : o == 5 ? args.f[5] + row1 : (o == 4 && nyq_z) ? aux_z : args.f[3] + row1;
#pragma unroll
        for (int j1 = 0; j1 < N1; ++j1) g[j1] = src[N2 * j1 + c1];
      }
      // v = conj(m g), m = cA ky^2 + cB ky + cC: whole numbers below 2^24, exact in FP32 (FP64
      // data convert the product once; the FP64 pipe is what bounds them)
      const float cA = o == 0 ? 1.f : 0.f;
      const float cB = o == 2 ? (nyq_z ? (float)(N / 2) : fz) : o == 3 ? 1.f : 0.f;
      const float cC = o == 1 ? fz * fz : o == 4 ? (nyq_z ? (float)(N / 2) : fz) : o == 5 ? 1.f : 0.f;
      const bool abs_y = nyq_z && o == 2;
      V v[N1];
      if (sizeof(T) == 8 && o == 5) {
#pragma unroll
        for (int j1 = 0; j1 < N1; ++j1) v[j1] = cconj(g[j1]);
      } else {
#pragma unroll
        for (int j1 = 0; j1 < N1; ++j1) {
          float fy = fc1 + (float)(N2 * j1 - (j1 >= N1 / 2 ? N : 0));
          if (j1 == N1 / 2 && c1 == 0) fy = (float)(N / 2);
          if (abs_y) fy = fabsf(fy);
          const T m = (T)((cA * fy + cB) * fy + cC);
          v[j1] = cmake<V>(m * g[j1].x, -m * g[j1].y);
        }
      }
      if (o == 3) {  // the k_x = N/2 term of H_xy takes the sign of ky
#pragma unroll
        for (int j1 = N1 / 2; j1 < N1; ++j1) {
          const T f2 = (T)(par * (fc1 + (float)(N2 * j1 - N)));
          const V a = aux_x[N2 * j1 + c1];
          v[j1].x += f2 * a.x;
          v[j1].y -= f2 * a.y;
        }
        if (c1 == 0) {  // ky = N/2: |k_x| (N/2) P
          const V b = aux_y[x0 + r1];
          v[N1 / 2] = cmake<V>((T)(N / 2) * b.x, -(T)(N / 2) * b.y);
        }
      }
      dft_regs<N1, N / N1>(v, s_tw);
      V* Tr = T1 + r1 * G::RS;
#pragma unroll
      for (int k1 = 0; k1 < N1; ++k1)
        Tr[k1 * (N2 + 1) + c1] = k1 == 0 ? v[k1] : cmul(v[k1], s_tw[k1 * N2 + c1]);
    }
    // With N1 == N2 a row's threads are the same in both stages and lie in one warp.  After this
    // point every thread that reads the rows this output overwrites has read them.
    if constexpr (N1 == N2 && !G::SPLIT) __syncwarp();
    else __syncthreads();
    V u[N2];
    const V* Tp = T1 + row * G::RS + lane * (N2 + 1);
#pragma unroll
    for (int j2 = 0; j2 < N2; ++j2) u[j2] = Tp[j2];
    dft_regs<N2, N / N2>(u, s_tw);
    V* dst = args.f[slot] + plane + (int64_t)(x0 + row) * N + lane;
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) dst[N1 * k2] = cconj(u[k2]);
  }
}

template <typename T, int N, int RB>
static void launch_yh(const YHessArgs<T>* a, int count, const vec2_t<T>* tw, cudaStream_t s) {
  using G = YHGeom<T, N>;
  raise_smem_limit<k_y_hessian<T, N, RB>>(G::SMEM);
  YHBatch<T, RB> yb;
  for (int r = 0; r < count; ++r) yb.a[r] = a[r];
  k_y_hessian<T, N, RB><<<dim3((N / 2 + 1) * (N / G::P), G::SPLIT ? 2 : 1, count),
                          dim3(G::THREADS, G::OUTS), G::SMEM, s>>>(yb, tw);
}

template <typename T, int N>
void launch_y_hessian(const YHessArgs<T>* a, int count, const vec2_t<T>* tw, cudaStream_t s) {
  if (count == 1) {
    launch_yh<T, N, 1>(a, 1, tw, s);
  } else if constexpr (sizeof(T) == 4 && N <= 128) {
    if (count > 1 && count <= kBatchMax) launch_yh<T, N, kBatchMax>(a, count, tw, s);
  }
}

#define DGP_INST_YH(T, N) \
  template void launch_y_hessian<T, N>(const YHessArgs<T>*, int, const vec2_t<T>*, cudaStream_t);
#define DGP_INST_YH_ALL(T) DGP_INST_YH(T, 16) DGP_INST_YH(T, 32) DGP_INST_YH(T, 48) DGP_INST_YH(T, 64) \
  DGP_INST_YH(T, 96) DGP_INST_YH(T, 128) DGP_INST_YH(T, 256) DGP_INST_YH(T, 512)
DGP_INST_YH_ALL(float)
DGP_INST_YH_ALL(double)

}  // namespace dgp
