// The relaxation pass with every row transformed inside one warp.
// Included by relax_tma.cu, which holds the arithmetic policies, the TMA helpers and the host side.
//
// A row is a pencil of the tile transforms of tile_slots.cuh (N2 lanes of a warp; the transpose of a
// field pair's N complex values in the N + 2 slots the row has in the pair's two tiles).  No other
// warp touches a row's slots, so the transforms need no block barrier (the version with a row's
// lanes spread over the CTA has 17 in a CTA); a copy into a used buffer is issued by whichever warp
// arrives last.
// The forward transform takes each row of D_new straight from registers as a real transform
// (N1 / 2 + 1 of the N1 stage-two columns are needed) and leaves the half spectrum in the same tile
// layout, which one TMA store per box writes out.
//
// What bounds it (256^3, 675 MB of algorithmic traffic, 135 us, 0.74 of the copy rate): instruction
// issue (about 63 % of the cycles) and the wait for a CTA's first tiles at 24 warps per SM.  Tried: CTAs
// that stay and take every gridDim-th tile, loading the next tile's first pair during the forward
// transform (153 us: the state carried from tile to tile spills at 80 registers, and two CTAs of 128
// are no faster); two CTAs of 128 registers (159 us).  512^3 holds one CTA of 8 warps per SM, of 227
// registers a thread (168 with pair arithmetic).
#pragma once

#include "tile_slots.cuh"

namespace dgp {

// Split of a row: that of the other passes, except that 48 takes four lanes of 12 samples and 96 eight
// lanes of 12 (rows of 3 or 6 lanes do not fill warps), with twiddles from the table of all W_N^t
// instead of the phase table of the other split.  At 96 the 12 columns of the second stage take two
// rounds of the 8 lanes, the second half empty, and D_new goes through shared memory to the lanes of
// the forward transform.  (Four lanes of 24 samples need 128 registers and leave 8 warps per SM to a
// single 96^3 mesh: 25 us against 22 for rows spread over the CTA.)
// WIDE: twice the lanes per row (96: the same), and after the second stage the values of a field pair
// go through the row's slots to all of them, N1 to a lane.
template <int N, bool WIDE> struct RowSplit {
  static constexpr int N1 = Split<N>::N1, N2 = Split<N>::N2;
  static constexpr bool PHASES = true;
};
template <> struct RowSplit<48, false> { static constexpr int N1 = 12, N2 = 4; static constexpr bool PHASES = false; };
template <> struct RowSplit<96, false> { static constexpr int N1 = 12, N2 = 8; static constexpr bool PHASES = false; };
template <> struct RowSplit<32, true> { static constexpr int N1 = 4, N2 = 8; static constexpr bool PHASES = false; };
template <> struct RowSplit<48, true> { static constexpr int N1 = 6, N2 = 8; static constexpr bool PHASES = false; };
template <> struct RowSplit<96, true> { static constexpr int N1 = 12, N2 = 8; static constexpr bool PHASES = false; };

template <int N, bool WIDE> struct RowGeom {
  static constexpr int N1 = RowSplit<N, WIDE>::N1, N2 = RowSplit<N, WIDE>::N2, Q = (N1 + N2 - 1) / N2;
  static constexpr bool EVEN = WIDE || N1 % N2 == 0;  // a lane ends with the samples of its column
  static constexpr int PTS = WIDE ? N1 : Q * N2;      // values of a lane after the inverse transform
  static constexpr int TY = 16, THREADS = TY * N2, WARPS = THREADS / 32;
  static constexpr int NK = N / 2 + 1;
  static constexpr int NBOX = (NK + 255) / 256;
  // lines per TMA box: whole swizzle periods when there are two (lines past the end read as zero
  // and are not stored)
  static constexpr int BOXK = NBOX == 1 ? NK : ((NK + NBOX - 1) / NBOX + 7) / 8 * 8;
  static constexpr int FIELD = (NBOX * BOXK * 128 + 1023) / 1024 * 1024;
  static constexpr int ROWP = N + N2;               // padded D and S rows (floats)
  static constexpr int DS = 2 * TY * ROWP * 4;
  // a field pair, or the rows of D and S
  static constexpr int BUF = 2 * FIELD > DS ? 2 * FIELD : (DS + 1023) / 1024 * 1024;
  static constexpr int EXTRA = 16 + 4 * 8 * WARPS + 16 + 32;  // barriers, partials, mean, counters
  static constexpr size_t SMEM = 1024 + 2 * BUF + N * 8 + EXTRA;
  // 24 warps per SM at 80 registers
  static constexpr int MINB = N == 512 ? 1 : 768 / THREADS;
};

// W_R^k, R dividing 32 or 24
template <int R> __device__ __forceinline__ float2 twiddle_r(int k) {
  if constexpr (32 % R == 0) return twiddle_c<float2, R>(k);
  else return twiddle24<float2>(24 / R * k);
}

// Real DFT of R values: X[0..R/2], X[0] and (R even) X[R/2] real.  Decimation in time.
template <int R>
__device__ __forceinline__ void rdft(const float (&x)[R], float2 (&X)[R / 2 + 1]) {
  if constexpr (R == 2) {
    X[0] = make_float2(x[0] + x[1], 0.f);
    X[1] = make_float2(x[0] - x[1], 0.f);
  } else if constexpr (R == 3) {
    const float h = 0.86602540378443864676f, s = x[1] + x[2];
    X[0] = make_float2(x[0] + s, 0.f);
    X[1] = make_float2(x[0] - 0.5f * s, -h * (x[1] - x[2]));
  } else {
    constexpr int H = R / 2;
    float e[H], o[H];
#pragma unroll
    for (int i = 0; i < H; ++i) {
      e[i] = x[2 * i];
      o[i] = x[2 * i + 1];
    }
    float2 E[H / 2 + 1], O[H / 2 + 1];
    rdft<H>(e, E);
    rdft<H>(o, O);
    X[0] = make_float2(E[0].x + O[0].x, 0.f);
    X[H] = make_float2(E[0].x - O[0].x, 0.f);
#pragma unroll
    for (int k = 1; 2 * k < H; ++k) {
      float2 t;
      if (8 * k == R) {
        const float c = 0.70710678118654752440f;
        t = make_float2((O[k].x + O[k].y) * c, (O[k].y - O[k].x) * c);
      } else {
        t = cmul(O[k], twiddle_r<R>(k));
      }
      X[k] = cadd(E[k], t);
      X[H - k] = cconj(csub(E[k], t));
    }
    if constexpr (H % 2 == 0) X[H / 2] = make_float2(E[H / 2].x, -O[H / 2].x);
  }
}

// W_N^{k1 c} of the four-step split from the table in shared memory
template <int N, bool WIDE> __device__ __forceinline__ float2 row_phase(const float2* s_tw, int k1, int c) {
  if constexpr (RowSplit<N, WIDE>::PHASES) return s_tw[k1 * RowSplit<N, WIDE>::N2 + c];
  else return s_tw[k1 * c];
}

// the row's slots: those from N / 2 on are in the second tile
template <int N, bool WIDE>
using RowSlots = TileSlots<RowGeom<N, WIDE>::N1, RowGeom<N, WIDE>::N2, RowGeom<N, WIDE>::FIELD - (N / 2) * 128>;

// First stage of the inverse z transform of the pair in buf, its transpose in the row's slots.
template <int N, bool WIDE>
__device__ __forceinline__ void row_pair_first(unsigned char* buf, const float2* s_tw, int r, int c) {
  using G = RowGeom<N, WIDE>;
  using S = RowSlots<N, WIDE>;
  constexpr int N1 = G::N1, N2 = G::N2;
  {
    float2 v[N1];
    const unsigned char* TA = buf;
    const unsigned char* TB = buf + G::FIELD;
    const int off_d = S::line(c, r), off_m = S::line(N - c, r);
#pragma unroll
    for (int j1 = 0; j1 < N1; ++j1) {
      // k = N2 j1 + c; beyond N / 2 the conjugate of line N - k
      bool mirror;
      if (j1 < N1 / 2) mirror = false;
      else if (j1 > N1 / 2) mirror = true;
      else mirror = c != 0;
      const int off = mirror ? S::sample(off_m, -j1) : S::sample(off_d, j1);
      float2 A = tile_at(TA, off), B = tile_at(TB, off);
      if (mirror) {
        A.y = -A.y;
        B.y = -B.y;
      } else if ((j1 == 0 || j1 == N1 / 2) && c == 0) {
        A.y = 0.f;
        B.y = 0.f;
      }
      v[j1] = make_float2(A.x - B.y, -(A.y + B.x));  // conj(A + i B)
    }
    __syncwarp();  // the row's values are read: its slots hold the transpose now
    dft_regs<N1, N / N1>(v, s_tw);
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1)
      tile_at(buf, S::by_col(off_d, k1)) = k1 == 0 ? v[k1] : cmul(v[k1], row_phase<N, WIDE>(s_tw, k1, c));
  }
  __syncwarp();
}

// The two fields (a, -b) of sample z = c + N2 i after row_pair_to_slots.
template <int N, bool WIDE>
__device__ __forceinline__ float2 row_pair_sample(const unsigned char* buf, int r, int c, int i) {
  return tile_at(buf, RowSlots<N, WIDE>::folded(c + RowGeom<N, WIDE>::N2 * i, r));
}

// Inverse z transform of the pair in buf: rows k1 on the lanes that have one, then sample z to the slot
// of line z.
template <int N, bool WIDE>
__device__ __forceinline__ void row_pair_to_slots(unsigned char* buf, const float2* s_tw, int r, int c) {
  using G = RowGeom<N, WIDE>;
  using S = RowSlots<N, WIDE>;
  constexpr int N1 = G::N1, N2 = G::N2, Q = G::Q;
  row_pair_first<N, WIDE>(buf, s_tw, r, c);
  float2 u[Q][N2];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    if (c + N2 * q >= N1) continue;
    const int base = S::by_row_base(c + N2 * q, r);
#pragma unroll
    for (int j2 = 0; j2 < N2; ++j2) u[q][j2] = tile_at(buf, S::by_row(base, j2));
    dft_regs<N2, N / N2>(u[q], s_tw);
  }
  __syncwarp();
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    if (c + N2 * q >= N1) continue;
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) tile_at(buf, S::folded(c + N2 * q + N1 * k2, r)) = u[q][k2];
  }
  __syncwarp();
}

// Inverse z transform of the pair in buf: on return a[i], b[i] with i = q + Q k2 are the two fields at
// z = k1 + N1 k2, k1 = c + N2 q (zero where k1 >= N1); z = c + N2 i when EVEN.
template <int N, bool WIDE>
__device__ __forceinline__ void row_pair_inverse(unsigned char* buf, const float2* s_tw, int r, int c,
                                                 float (&a)[RowGeom<N, WIDE>::PTS], float (&b)[RowGeom<N, WIDE>::PTS]) {
  using G = RowGeom<N, WIDE>;
  using S = RowSlots<N, WIDE>;
  constexpr int N1 = G::N1, N2 = G::N2, Q = G::Q;
  if constexpr (WIDE) {
    row_pair_to_slots<N, WIDE>(buf, s_tw, r, c);
#pragma unroll
    for (int i = 0; i < N1; ++i) {
      const float2 v = row_pair_sample<N, WIDE>(buf, r, c, i);
      a[i] = v.x;
      b[i] = -v.y;
    }
    return;
  }
  row_pair_first<N, WIDE>(buf, s_tw, r, c);
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    if (!G::EVEN && c + N2 * q >= N1) {
#pragma unroll
      for (int k2 = 0; k2 < N2; ++k2) a[q + Q * k2] = b[q + Q * k2] = 0.f;
      continue;
    }
    const int base = S::by_row_base(c + N2 * q, r);
    float2 u[N2];
#pragma unroll
    for (int j2 = 0; j2 < N2; ++j2) u[j2] = tile_at(buf, S::by_row(base, j2));
    dft_regs<N2, N / N2>(u, s_tw);
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) {
      a[q + Q * k2] = u[k2].x;
      b[q + Q * k2] = -u[k2].y;
    }
  }
}

// Forward z transform of the row whose values at z = c + N2 j1 are d[j1]; the half spectrum goes to
// the first tile of buf in the tile layout (line kz, row r).
template <int N, bool WIDE>
__device__ __forceinline__ void row_forward(unsigned char* buf, const float2* s_tw, int r, int c,
                                            const float (&d)[RowGeom<N, WIDE>::N1]) {
  using G = RowGeom<N, WIDE>;
  using S = RowSlots<N, WIDE>;
  constexpr int N1 = G::N1, N2 = G::N2;
  {
    float2 V[N1 / 2 + 1];
    rdft<N1>(d, V);
    const int base = S::line(c, r);
#pragma unroll
    for (int k1 = 0; k1 <= N1 / 2; ++k1) {
      const float2 w = row_phase<N, WIDE>(s_tw, k1, c);
      const float2 t = k1 == 0 ? V[0] : k1 == N1 / 2 ? make_float2(V[k1].x * w.x, V[k1].x * w.y) : cmul(V[k1], w);
      tile_at(buf, S::by_col(base, k1)) = t;
    }
  }
  __syncwarp();
  // columns k1 = 0 .. N1 / 2: one round, and a second for those from N2 on (k1 = N1 / 2 alone where
  // N1 = 2 N2, k1 = 4 .. 6 at 48 = 12 x 4)
  constexpr int ROUNDS = (N1 / 2) / N2 + 1;
  float2 u[ROUNDS][N2];
#pragma unroll
  for (int q = 0; q < ROUNDS; ++q) {
    const int k1 = c + N2 * q;
    if (k1 <= N1 / 2) {
      const int base = S::by_row_base(k1, r);
#pragma unroll
      for (int j2 = 0; j2 < N2; ++j2) u[q][j2] = tile_at(buf, S::by_row(base, j2));
    }
  }
  __syncwarp();  // all columns of the row are read: its lines may be written
#pragma unroll
  for (int q = 0; q < ROUNDS; ++q) {
    const int k1 = c + N2 * q;
    if (k1 <= N1 / 2) {
      dft_regs<N2, N / N2>(u[q], s_tw);
#pragma unroll
      for (int k2 = 0; k2 < N2; ++k2) {
        const int k = k1 + N1 * k2;
        const bool mirror = k > N / 2;
        // the columns k1 = 0 and N1 / 2 are their own mirror images
        if (mirror && (k1 == 0 || k1 == N1 / 2)) continue;
        const int kz = mirror ? N - k : k;
        const float2 o = mirror ? cconj(u[q][k2]) : u[q][k2];
        tile_at(buf, S::line(kz, r)) = o;
      }
    }
  }
}

// Whether a pass takes the wide rows: FP64 arithmetic always (it is what the pass waits for: an FP64
// instruction holds a quarter of the SM for some 60 cycles, at 32^3 and 48^3 there are too few warps for
// 8 and 12 points a lane, at 96^3 a third of the lanes would idle; per solve of 23-26 evaluations 837 ->
// 728, 1094 -> 904 and 3043 -> 2535 us), float pairs and any arithmetic at 48^3 where one mesh does not
// fill the chip (float pairs at 32, 48, 96: 681 -> 636, 844 -> 759, 1333 -> 1284 us; FP32 at 48^3 766 ->
// 737).  FP32 at 32^3 gains nothing, at 96^3 it loses (1154 -> 1236: the trip through the slots).
template <int N, class AR, int RB> struct RowWide {
  static constexpr bool F64 = std::is_same<typename AR::Sum, double>::value;
  static constexpr bool EFT = std::is_same<AR, RxEFT>::value;
  static constexpr bool W = (N == 32 || N == 48 || N == 96) && (F64 || (RB == 1 && (EFT || N == 48)));
  // Float pairs at 512^3, 32 points to a lane: unrolled over them the arithmetic alone is some 56 KB of
  // code, which 8 warps an SM wait for.  The points go in a rolled loop then, their fields through the row's
  // slots and the accumulators through shared memory: 3989 -> 2335 us a launch (2523 with rows spread over
  // the CTA).
  static constexpr bool ROLL = N == 512 && EFT;
  using G = RowGeom<N, W>;
  static constexpr size_t SMEM = G::SMEM + (ROLL ? sizeof(float2) * G::THREADS * G::PTS : 0);
};

template <int N, class AR, int RB>
__global__ void __launch_bounds__(RowGeom<N, RowWide<N, AR, RB>::W>::THREADS, RowGeom<N, RowWide<N, AR, RB>::W>::MINB)
    k_relax_rows(const __grid_constant__ RelaxTmaBatch<RB> batch, const float2* __restrict__ g_tw) {
  const RelaxTmaArgs& args = batch.a[RB > 1 ? blockIdx.z : 0];  // realisation of this CTA
  if (args.skip && *args.skip) return;
  constexpr bool WIDE = RowWide<N, AR, RB>::W, ROLL = RowWide<N, AR, RB>::ROLL;
  using G = RowGeom<N, WIDE>;
  using Acc = typename AR::Acc;
  using Sum = typename AR::Sum;
  constexpr int N1 = G::N1, N2 = G::N2, TY = G::TY, ROWP = G::ROWP, WARPS = G::WARPS;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* buf0 = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* buf1 = buf0 + G::BUF;
  float2* s_tw = reinterpret_cast<float2*>(buf1 + G::BUF);
  uint64_t* bars = reinterpret_cast<uint64_t*>(s_tw + N);        // [2]
  double* s_part = reinterpret_cast<double*>(bars + 2);          // [4][WARPS]
  double* s_mean = s_part + 4 * WARPS;                           // mean, then its float pair
  // arrivals (A read, B read, done), then flags: a wait gave up, C issued, the rows issued
  int* s_cnt = reinterpret_cast<int*>(s_mean + 2);
  const int tid = threadIdx.x, wid = tid >> 5, wl = tid & 31;
  const int c = (wl >> 1) % N2, r = wid * (32 / N2) + 2 * ((wl >> 1) / N2) + (wl & 1);
  const int x = blockIdx.y, y0 = blockIdx.x * TY;
  const RelaxParams& rp = args.rp;
  const uint64_t lim = args.wait_ns;

  auto issue = [&](unsigned char* dst, int fa, int fb, uint64_t* bar) {
    mbar_expect_tx(bar, 2u * G::NBOX * G::BOXK * 128u);
#pragma unroll
    for (int b = 0; b < G::NBOX; ++b) {
      tma_load_3d(dst + b * G::BOXK * 128, &args.map[fa], 2 * y0, x, b * G::BOXK, bar);
      tma_load_3d(dst + G::FIELD + b * G::BOXK * 128, &args.map[fb], 2 * y0, x, b * G::BOXK, bar);
    }
  };
  if (tid == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&bars[1], 1);
    mbar_init_fence();
    // pair A = (H_xy, H_xz) -> buf0, pair B = (H_yz, N) -> buf1 (phase 0 of each barrier)
    if (!args.withhold) issue(buf0, 2, 3, &bars[0]);
    issue(buf1, 4, 5, &bars[1]);
    const double m = args.dsum ? args.dsum[0] * rp.inv_m : 0.0;
    s_mean[0] = m;
    float* mp = reinterpret_cast<float*>(s_mean + 1);
    mp[0] = (float)m;
    mp[1] = (float)(m - (double)mp[0]);
    for (int i = 0; i < 6; ++i) s_cnt[i] = 0;
  }
  for (int i = tid; i < N; i += G::THREADS) s_tw[i] = g_tw[(RowSplit<N, WIDE>::PHASES ? N : 0) + i];
  __syncthreads();
  const double mean = s_mean[0];
  const float m_hi = reinterpret_cast<const float*>(s_mean + 1)[0];
  const float m_lo = reinterpret_cast<const float*>(s_mean + 1)[1];

  // A wait that gives up records the fault (the solve then ends with DGP_E_TIMEOUT and its outputs
  // are discarded); the warp goes on without waiting again and no further copy is issued.
  bool ok = true;
  auto wait = [&](uint64_t* bar, unsigned parity) {
    if (ok && !mbar_wait_bounded(bar, parity, lim)) {
      ok = false;
      atomicExch(args.fault, 1);
      *reinterpret_cast<volatile int*>(&s_cnt[3]) = 1;
    }
    ok = __all_sync(0xffffffffu, ok);
  };
  // true in the last warp to arrive; orders the warps' accesses before what it issues
  auto last_warp = [&](int k) {
    fence_proxy_async();
    __syncwarp();
    int last = 0;
    if (wl == 0) {
      __threadfence_block();
      last = atomicAdd(&s_cnt[k], 1) == WARPS - 1;
      __threadfence_block();
    }
    return __shfl_sync(0xffffffffu, last, 0) != 0;
  };
  auto gave_up = [&]() { return *reinterpret_cast<volatile int*>(&s_cnt[3]) != 0; };

  constexpr int PTS = G::PTS, Q = G::Q, HELD = ROLL ? 1 : PTS;
  Acc acc[HELD];
  float ra[HELD], rb[HELD];
  // ROLL: the thread's accumulators, [point][thread]
  float2* s_acc = reinterpret_cast<float2*>(s_cnt + 8) + tid;
  wait(&bars[0], 0);
  if constexpr (ROLL) {
    row_pair_to_slots<N, WIDE>(buf0, s_tw, r, c);
#pragma unroll 4
    for (int i = 0; i < PTS; ++i) {
      const float2 v = row_pair_sample<N, WIDE>(buf0, r, c, i);
      AR::pair_a(acc[0], v.x, -v.y);
      s_acc[i * G::THREADS] = make_float2(acc[0].hi, acc[0].lo);
    }
  } else {
    row_pair_inverse<N, WIDE>(buf0, s_tw, r, c, ra, rb);
#pragma unroll
    for (int i = 0; i < PTS; ++i) AR::pair_a(acc[i], ra[i], rb[i]);
  }
  if (last_warp(0) && wl == 0 && !gave_up()) {  // pair C, the diagonal
    s_cnt[4] = 1;
    issue(buf0, 0, 1, &bars[0]);
  }
  wait(&bars[1], 0);
  if constexpr (ROLL) {
    row_pair_to_slots<N, WIDE>(buf1, s_tw, r, c);
#pragma unroll 4
    for (int i = 0; i < PTS; ++i) {
      const float2 v = row_pair_sample<N, WIDE>(buf1, r, c, i), t = s_acc[i * G::THREADS];
      acc[0] = Acc{t.x, t.y};
      AR::pair_b(acc[0], v.x, -v.y, rp);
      s_acc[i * G::THREADS] = make_float2(acc[0].hi, acc[0].lo);
    }
  } else {
    row_pair_inverse<N, WIDE>(buf1, s_tw, r, c, ra, rb);
#pragma unroll
    for (int i = 0; i < PTS; ++i) AR::pair_b(acc[i], ra[i], rb[i], rp);
  }
  float* sD = reinterpret_cast<float*>(buf1);
  float* sS = sD + TY * ROWP;
  const int64_t rbase0 = ((int64_t)x * N + y0) * N;
  // the rows of D and S; the flag may be set meanwhile, so one answer for the warp
  if (last_warp(1) && !__any_sync(0xffffffffu, gave_up())) {
    if (wl == 0) {
      s_cnt[5] = 1;
      mbar_expect_tx(&bars[1], 2u * TY * N * 4);
    }
    __syncwarp();
    const float* src = (wl < TY ? args.D : args.S) + rbase0 + (int64_t)(wl % TY) * N;
    bulk_load((wl < TY ? sD : sS) + (wl % TY) * ROWP, src, N * 4, &bars[1]);
  }
  wait(&bars[0], 1);
  // a, b: two diagonal second derivatives
  if constexpr (ROLL) row_pair_to_slots<N, WIDE>(buf0, s_tw, r, c);
  else row_pair_inverse<N, WIDE>(buf0, s_tw, r, c, ra, rb);
  wait(&bars[1], 1);
  Sum rsum{};
  FP acc_d{0.f, 0.f};  // sum of D_new: its mean is removed next iteration
  float nbad = 0.f, nonfin = 0.f;
  float* dst = args.Dnew + rbase0 + (int64_t)r * N;
  // residual and update at sample z, which returns D_new
  auto update = [&](Acc& t, float fa, float fb, int z) {
    const PointOut o = AR::finish(t, fa, fb, sD[r * ROWP + z], sS[r * ROWP + z], m_hi, m_lo, mean, rp, rsum, nonfin);
    float bpt = o.bp, dt = o.dt;
    if (o.neg) {
      nbad += 1.f;
      bpt = rp.bad_bp_f;
      dt = 0.f;
    }
    float dn;
    if constexpr (AR::kApproxRoot) {
      // D_new is an FP32 datum: the hardware square root and the full-range division (a few
      // ulp, far below the FFTs' rounding of the fields it is computed from)
      dn = fdiv_full(2.f * bpt, rp.alpha_f + sqrt_approx(dt));
    } else {
      dn = 2.f * bpt / (rp.alpha_f + sqrtf(dt));
    }
    dst[z] = dn;
    if constexpr (std::is_same<AR, RxF32>::value) acc_d.hi += dn;
    else fp_acc(acc_d, FP{dn, 0.f});
    return dn;
  };
  constexpr bool VIA_SD = ROLL || !G::EVEN;  // D_new reaches the forward transform's lanes through sD
  if constexpr (ROLL) {
#pragma unroll 2
    for (int i = 0; i < PTS; ++i) {
      const float2 v = row_pair_sample<N, WIDE>(buf0, r, c, i), t = s_acc[i * G::THREADS];
      acc[0] = Acc{t.x, t.y};
      const int z = c + N2 * i;
      sD[r * ROWP + z] = update(acc[0], v.x, -v.y, z);
    }
  } else {
#pragma unroll
    for (int i = 0; i < PTS; ++i) {
      const int k1 = c + N2 * (i % Q);
      if (!G::EVEN && k1 >= N1) continue;
      const int z = G::EVEN ? c + N2 * i : k1 + N1 * (i / Q);
      const float dn = update(acc[i], ra[i], rb[i], z);
      if constexpr (VIA_SD) sD[r * ROWP + z] = dn;
      else ra[i] = dn;
    }
  }
  __syncwarp();  // the row's slots of buf0 are read, its D_new is written
  if constexpr (!VIA_SD) {
    row_forward<N, WIDE>(buf0, s_tw, r, c, ra);
  } else {
    float d[N1];
#pragma unroll
    for (int j1 = 0; j1 < N1; ++j1) d[j1] = sD[r * ROWP + N2 * j1 + c];
    row_forward<N, WIDE>(buf0, s_tw, r, c, d);
  }
  // ---- statistics: within a warp float pairs (FP64 for the FP64 policy), across warps FP64
  if constexpr (std::is_same<Sum, double>::value) {
    double v4[4] = {rsum, (double)acc_d.hi + (double)acc_d.lo, (double)nbad, (double)nonfin};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v4[k] += __shfl_xor_sync(0xffffffffu, v4[k], o);
      if (wl == 0) s_part[k * WARPS + wid] = v4[k];
    }
  } else {
    FP r2 = pair_of(rsum), d2 = acc_d;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      fp_acc(r2, FP{__shfl_xor_sync(0xffffffffu, r2.hi, o), __shfl_xor_sync(0xffffffffu, r2.lo, o)});
      fp_acc(d2, FP{__shfl_xor_sync(0xffffffffu, d2.hi, o), __shfl_xor_sync(0xffffffffu, d2.lo, o)});
    }
    const unsigned nb = __reduce_add_sync(0xffffffffu, (unsigned)nbad);
    const unsigned nf = __reduce_add_sync(0xffffffffu, (unsigned)nonfin);
    if (wl == 0) {
      s_part[0 * WARPS + wid] = (double)r2.hi + (double)r2.lo;
      s_part[1 * WARPS + wid] = (double)d2.hi + (double)d2.lo;
      s_part[2 * WARPS + wid] = (double)nb;
      s_part[3 * WARPS + wid] = (double)nf;
    }
  }
  if (!last_warp(2)) return;
  if (wl < 4) {
    double t = 0.0;
    for (int w = 0; w < WARPS; ++w) t += *reinterpret_cast<volatile double*>(&s_part[wl * WARPS + w]);
    args.partials[((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * 4 + wl] = t;
  }
  if (wl == 0) {
    if (gave_up()) {
      // every copy issued lands, or this wait runs out too, before the CTA's shared memory is given back:
      // C and the rows are issued only once the phase before them has completed (bounded; nothing waits
      // for a copy that was not issued)
      const uint64_t lim2 = 4 * lim + 1000000000ull;
      if (s_cnt[4]) mbar_wait_bounded(&bars[0], 1, lim2);
      else if (!args.withhold) mbar_wait_bounded(&bars[0], 0, lim2);
      mbar_wait_bounded(&bars[1], s_cnt[5] ? 1 : 0, lim2);
      return;
    }
#pragma unroll
    for (int b = 0; b < G::NBOX; ++b) tma_store_3d(&args.out_map, 2 * y0, x, b * G::BOXK, buf0 + b * G::BOXK * 128);
    bulk_store_wait();
  }
}

}  // namespace dgp
