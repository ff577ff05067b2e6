// Plane-resident Hessian pass for small meshes (FP32 data, realisations of one class).
//
// One CTA owns one kz plane of one realisation.  It reads the plane of the z spectrum of
// the iterate D (layout S[kz][x][y]) once, transforms it forward along y and along x in
// shared memory, and for each of the six outputs of the relaxation (H_yy, H_zz, H_xy, H_xz,
// H_yz and N, Sec. III.B: nabla_ij C(k) = -k_i k_j C(k), sqrt(-lapbar) C = -D / kbar)
// forms the multiplier, transforms back along x and y and writes the plane of the output
// (kz, x, y), ready for the relaxation pass's inverse z transform.  The y and z wavenumbers commute
// with the x inverse, so the x inverse runs three times, not six: of P = D / k^2 (then times k_y^2,
// k_z^2 and k_y k_z for H_yy, H_zz and H_yz; H_xx is the trace's rest), of k_x P (H_xy, H_xz) and of N.  This replaces the
// y pass of D_new, the Hessian x pass and the six-field inverse y pass of an iteration: per
// iteration the six output spectra cross HBM once (written here, read by the relaxation)
// instead of three times.  A plane of N x N complex floats must fit three times in shared
// memory (the spectrum, its x inverse, an output), so the pass serves N <= 96.
//
// Transforms are the four-step split N = N1 * N2 done in place on a line of the plane:
// forward, stage 1 takes the N1 elements N2*j1 + j2 of a line, transforms them, multiplies
// by W_N^{j2 k1} and puts them back at N2*k1 + j2; stage 2 transforms the N2 contiguous
// elements N2*k1 + j2 (j2 < N2) and leaves X[k1 + N1*k2] at position N2*k1 + k2 (digit
// order).  The inverse runs the stages in the opposite order, from digit order back to
// natural order, as conj(DFT(conj(.))).  The plane's row pitch is N + 1 (odd): within a
// stage consecutive threads take consecutive lines of the same stage index, so a half-warp
// touches 16 different banks along either axis.
#include <type_traits>

#include "fft_core.cuh"
#include "kernels.cuh"

namespace dgp {

template <int N> struct PGeom {
  static constexpr int N1 = Split<N>::N1, N2 = Split<N>::N2;
  static constexpr int PITCH = N + 1;
  static constexpr int PLANE = N * PITCH;  // complex elements of one plane buffer
  static constexpr int THREADS = N == 96 ? 768 : N == 64 ? 256 : N == 48 ? 192 : N == 32 ? 128 : 64;
  static constexpr int MINB = N == 96 ? 1 : N == 64 ? 2 : N == 48 ? 4 : N == 32 ? 4 : 8;
  static constexpr size_t SMEM = sizeof(float2) * ((size_t)3 * PLANE + N);
  static_assert(N % 16 == 0 || N < 16, "lines of a stage are taken 16 at a time");
};

// Forward stage 1 on the lines of a plane buffer: line stride LS, element stride ES.
template <int N, int LS, int ES>
__device__ __forceinline__ void fwd_stage1(float2* __restrict__ b, const float2* __restrict__ s_tw) {
  using G = PGeom<N>;
  constexpr int N1 = G::N1, N2 = G::N2;
#pragma unroll 1
  for (int q = threadIdx.x; q < N * N2; q += G::THREADS) {
    const int line = q % N, j2 = q / N;
    float2* L = b + line * LS;
    float2 v[N1];
#pragma unroll
    for (int j1 = 0; j1 < N1; ++j1) v[j1] = L[(N2 * j1 + j2) * ES];
    dft_regs<N1, N / N1>(v, s_tw);
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) L[(N2 * k1 + j2) * ES] = k1 == 0 ? v[k1] : cmul(v[k1], s_tw[k1 * N2 + j2]);
  }
}

// Forward stage 2; MUL(line, k1, k2, value) may scale each output before it is stored.
template <int N, int LS, int ES, class Mul>
__device__ __forceinline__ void fwd_stage2(float2* __restrict__ b, const float2* __restrict__ s_tw, Mul mul) {
  using G = PGeom<N>;
  constexpr int N1 = G::N1, N2 = G::N2;
#pragma unroll 1
  for (int q = threadIdx.x; q < N * N1; q += G::THREADS) {
    const int line = q % N, k1 = q / N;
    float2* L = b + line * LS + N2 * k1 * ES;
    float2 u[N2];
#pragma unroll
    for (int j2 = 0; j2 < N2; ++j2) u[j2] = L[j2 * ES];
    dft_regs<N2, N / N2>(u, s_tw);
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) L[k2 * ES] = mul(line, k1, k2, u[k2]);
  }
}

// Inverse stage 1 from src (digit order) into dst: CONJ_IN conjugates on entry, and
// MUL(line, k1, k2, value) forms the input (a k-space multiplier) as it is read.  LINES lines; line N
// (the padding column) reads the line `extra` of src.
template <int N, int LS, int ES, bool CONJ_IN, int LINES, class Mul>
__device__ __forceinline__ void inv_stage1(const float2* src, float2* dst,  // may be the same buffer
                                           const float2* __restrict__ s_tw, int extra, Mul mul) {
  using G = PGeom<N>;
  constexpr int N1 = G::N1, N2 = G::N2;
#pragma unroll 1
  for (int q = threadIdx.x; q < LINES * N1; q += G::THREADS) {
    const int line = q % LINES, k1 = q / LINES;
    const int o = line * LS + N2 * k1 * ES;
    const int so = (LINES > N && line == N ? extra : line) * LS + N2 * k1 * ES;
    float2 u[N2];
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) {
      const float2 x = mul(line, k1, k2, src[so + k2 * ES]);
      u[k2] = CONJ_IN ? cconj(x) : x;
    }
    dft_regs<N2, N / N2>(u, s_tw);
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) dst[o + n2 * ES] = n2 == 0 ? u[n2] : cmul(u[n2], s_tw[k1 * N2 + n2]);
  }
}

// Inverse stage 2 in place, natural order out; CONJ_OUT conjugates on exit.
template <int N, int LS, int ES, bool CONJ_OUT, int LINES>
__device__ __forceinline__ void inv_stage2(float2* __restrict__ b, const float2* __restrict__ s_tw) {
  using G = PGeom<N>;
  constexpr int N1 = G::N1, N2 = G::N2;
#pragma unroll 1
  for (int q = threadIdx.x; q < LINES * N2; q += G::THREADS) {
    const int line = q % LINES, n2 = q / LINES;
    float2* L = b + line * LS;
    float2 w[N1];
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) w[k1] = L[(N2 * k1 + n2) * ES];
    dft_regs<N1, N / N1>(w, s_tw);
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1) L[(N2 * n1 + n2) * ES] = CONJ_OUT ? cconj(w[n1]) : w[n1];
  }
}

template <int RB> struct PlaneBatch {
  PlaneArgs a[RB];
};

// Plane <-> shared-memory copies (row pitch PITCH): TY rows of N at a time when the CTA's
// threads divide into whole rows, so no thread divides its index by N per element.
template <int N, bool TO_SMEM>
__device__ __forceinline__ void copy_plane(float2* __restrict__ sm, float2* __restrict__ g) {
  using G = PGeom<N>;
  if constexpr (G::THREADS % N == 0) {
    constexpr int RPI = G::THREADS / N;  // rows per round
    const int col = threadIdx.x % N, r0 = threadIdx.x / N;
#pragma unroll 4
    for (int r = r0; r < N; r += RPI) {
      if (TO_SMEM) sm[r * G::PITCH + col] = g[r * N + col];
      else g[r * N + col] = sm[r * G::PITCH + col];
    }
  } else {
    for (int i = threadIdx.x; i < N * N; i += G::THREADS) {
      if (TO_SMEM) sm[(i / N) * G::PITCH + i % N] = g[i];
      else g[i] = sm[(i / N) * G::PITCH + i % N];
    }
  }
}

template <int N, int RB>
__global__ void __launch_bounds__(PGeom<N>::THREADS, PGeom<N>::MINB)
    k_plane_hessian(const __grid_constant__ PlaneBatch<RB> pb, const float2* __restrict__ g_tw) {
  using G = PGeom<N>;
  constexpr int N1 = G::N1, N2 = G::N2, PITCH = G::PITCH;
  const PlaneArgs& args = pb.a[RB > 1 ? blockIdx.y : 0];
  if (args.skip && *args.skip) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* A = reinterpret_cast<float2*>(smem_raw);  // the spectrum of D, then P = D / k^2
  float2* B = A + G::PLANE;                          // one x inverse at a time
  float2* C = B + G::PLANE;                          // one output at a time
  float2* s_tw = C + G::PLANE;                       // the phase table
  for (int i = threadIdx.x; i < N; i += G::THREADS) s_tw[i] = g_tw[N + i];
  const int kz = blockIdx.x;
  copy_plane<N, true>(A, const_cast<float2*>(args.in) + (int64_t)kz * N * N);
  __syncthreads();
  // forward along y (lines = rows x), then along x (lines = columns)
  fwd_stage1<N, PITCH, 1>(A, s_tw);
  __syncthreads();
  auto keep = [](int, int, int, float2 v) { return v; };
  fwd_stage2<N, PITCH, 1>(A, s_tw, keep);
  __syncthreads();
  fwd_stage1<N, 1, PITCH>(A, s_tw);
  __syncthreads();
  // column py holds ky = k1y + N1 k2y at py = N2 k1y + k2y; the x stage 2 output of (k1, k2)
  // is kx = k1 + N1 k2.  Scale by 1 / (|n|^2 N^3) there (0 at k = 0).
  const KParams& kp = args.kp;
  const float inv_m = kp.inv_m_f;
  const bool nyq_z = kz == N / 2;
  const float fz = (float)(nyq_z ? -(N / 2) : kz);
  auto ky_of = [](int py) { return py / N2 + N1 * (py % N2); };
  auto scale = [&](int py, int k1, int k2, float2 v) {
    const float fx = (float)signed_index(k1 + N1 * k2, N), fy = (float)signed_index(ky_of(py), N);
    const float n2 = fx * fx + fy * fy + fz * fz;
    return cscale(v, n2 != 0.f ? inv_m / n2 : 0.f);
  };
  fwd_stage2<N, 1, PITCH>(A, s_tw, scale);
  __syncthreads();
  const float ikf = kp.local_only ? 0.f : 1.f / kp.kbkf_f;
  constexpr int PYN = N2 * ((N / 2) % N1) + (N / 2) / N1;  // digit-order place of index N / 2 on either axis
  // x inverses g: 0 P, 1 k_x P (k_x = +N/2 on its Nyquist index; the padding column carries |k_x| P of the
  // column k_y = N/2), 2 |k_x| P (the plane k_z = N/2 only), 3 N.  Outputs from each: 0 H_yy, 1 H_zz,
  // 4 H_yz; 2 H_xy, 3 H_xz; H_xz; 5 N.  Off-diagonal pairs take |k_i k_j| on a Nyquist index.
  // the y inverse of an output formed from B by ymul (rows x; the x inverse left its result
  // conjugated), and its store
  auto output = [&](int o, auto ymul) {
    inv_stage1<N, PITCH, 1, false, N>(B, C, s_tw, 0, ymul);
    __syncthreads();
    inv_stage2<N, PITCH, 1, true, N>(C, s_tw);
    __syncthreads();
    copy_plane<N, false>(C, args.out.p[o] + (int64_t)kz * N * N);
    __syncthreads();
  };
  // multiplier (cA k_y + cB) k_y + cC with k_y = +N/2 on its Nyquist index
  auto linear = [&](int o, float cA, float cB, float cC) {
    output(o, [&](int, int k1, int k2, float2 v) {
      float fy = (float)signed_index(k1 + N1 * k2, N);
      if (k1 + N1 * k2 == N / 2 || (nyq_z && o == 4)) fy = fabsf(fy);
      return cscale(v, (cA * fy + cB) * fy + cC);
    });
  };
  const float afz = fabsf(fz);
  auto group = [&](auto gc) {
    constexpr int g = decltype(gc)::value;
    constexpr int LINES = g == 1 ? N + 1 : N;
    inv_stage1<N, 1, PITCH, true, LINES>(A, B, s_tw, PYN, [&](int py, int k1, int k2, float2 v) {
      const int kx = k1 + N1 * k2;
      const float fx = (float)signed_index(kx, N);
      if constexpr (g == 0) return v;
      if constexpr (g == 1) return cscale(v, (py == N || kx == N / 2) ? fabsf(fx) : fx);
      if constexpr (g == 2) return cscale(v, fabsf(fx));
      const float fy = (float)signed_index(ky_of(py), N);
      return cscale(v, -sqrtf(fx * fx + fy * fy + fz * fz) * ikf);
    });
    __syncthreads();
    inv_stage2<N, 1, PITCH, false, LINES>(B, s_tw);
    __syncthreads();
    if constexpr (g == 0) {
#pragma unroll 1
      for (int j = 0; j < 3; ++j) linear(j == 2 ? 4 : j, j == 0 ? 1.f : 0.f, j == 2 ? afz : 0.f, j == 1 ? fz * fz : 0.f);
    } else if constexpr (g == 1) {
      output(2, [&](int x, int k1, int k2, float2 v) {
        const int ky = k1 + N1 * k2;
        const float fy = (float)signed_index(ky, N);
        if (ky == N / 2) return cscale(B[x * PITCH + N], (float)(N / 2));
        if (ky > N / 2) {  // the k_x = N/2 term takes the sign of k_y: subtract it twice
          const float2 a = A[PYN * PITCH + N2 * k1 + k2];
          const float c = x & 1 ? (float)N : -(float)N;
          v = make_float2(v.x + c * a.x, v.y - c * a.y);
        }
        return cscale(v, fy);
      });
      if (!nyq_z) linear(3, 0.f, 0.f, afz);
    } else {
      linear(g == 2 ? 3 : 5, 0.f, 0.f, g == 2 ? afz : 1.f);
    }
  };
  group(std::integral_constant<int, 0>{});
  group(std::integral_constant<int, 1>{});
  if (nyq_z) group(std::integral_constant<int, 2>{});
  group(std::integral_constant<int, 3>{});
}

template <int N>
static void launch_plane(const PlaneArgs* a, int count, const float2* tw, cudaStream_t s) {
  using G = PGeom<N>;
  PlaneBatch<kBatchMax> pb;
  for (int r = 0; r < count; ++r) pb.a[r] = a[r];
  raise_smem_limit<k_plane_hessian<N, kBatchMax>>(G::SMEM);
  k_plane_hessian<N, kBatchMax><<<dim3((unsigned)(N / 2 + 1), (unsigned)count), G::THREADS, G::SMEM, s>>>(pb, tw);
}

bool plane_hessian_supported(int n) { return n == 16 || n == 32 || n == 48 || n == 64 || n == 96; }

void launch_plane_hessian_batch(int n, const PlaneArgs* a, int count, const float2* tw, cudaStream_t s) {
  if (count < 1 || count > kBatchMax) return;
  switch (n) {
    case 16: launch_plane<16>(a, count, tw, s); break;
    case 32: launch_plane<32>(a, count, tw, s); break;
    case 48: launch_plane<48>(a, count, tw, s); break;
    case 64: launch_plane<64>(a, count, tw, s); break;
    case 96: launch_plane<96>(a, count, tw, s); break;
    default: break;
  }
}

}  // namespace dgp
