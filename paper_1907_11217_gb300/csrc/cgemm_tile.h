// Tiled complex64 product on CUDA cores (part of k_gemm_simt.cu: included
// inside its anonymous namespace). FP32 ALU-bound for large K, HBM-bound for
// many small products.
//
// A thread holds TM x TN outputs; every complex multiply-add is four FMAs in
// the order re += ax bx, re -= ay by (im likewise), k ascending. What bounds
// it is issue slots: 32 outputs a thread take 128 FMAs and six 16-byte shared
// loads per k (two rows of A or two columns of B each; a warp covers 8 x 4
// threads, so a load reads at most 128 different bytes). The two-wide
// fma.rn.f32x2 form (half the FMA issue slots, the same peak rate: 78 against
// 80 TF/s on independent chains) needs A pre-expanded as (ax, ax, -ay, ay) or
// expanded in registers, and measured slower either way (375 and 467 us where
// this takes 308: b16 M2048 N256 K256). Registers matter more than warps:
// three blocks of 64 x 64 at 150 registers a thread beat four at 128.
// Rows are padded by two elements, so the staging stores (a thread has two k
// of a row) fall in different banks. The next K tile is loaded into registers
// while the present one is multiplied (two shared buffers, one barrier a
// tile). Small tiles go NB to a block (consecutive tiles, of any product).
template <int BM, int BN, int TM, int TN, int BK, int NB>
struct TileCfg {
  static constexpr int TX = BN / TN, TY = BM / TM;
  static constexpr int NG = TX * TY;       // threads per product
  static constexpr int NT = NG * NB;
  static constexpr int CA = BM * BK / 2, CB = BN * BK / 2;  // 16-byte chunks (two k of a row)
  static constexpr int PA = (CA + NG - 1) / NG, PB = (CB + NG - 1) / NG;
};

// vec: rows of A and B start on 16 bytes (K even, bases and strides aligned)
template <int BM, int BN, int TM, int TN, int BK, int NB, int MINB>
__global__ void __launch_bounds__((BM / TM) * (BN / TN) * NB, MINB)
    cgemm_tile_kernel(const float2 *__restrict__ A, const float2 *__restrict__ B, float2 *__restrict__ C,
                      int64_t batch, int64_t M, int64_t N, int64_t K, int64_t sA, int64_t sB, int64_t sC,
                      const __grid_constant__ CScatter sc, int scatter, int vec, int64_t mt, int64_t nt) {
  using T = TileCfg<BM, BN, TM, TN, BK, NB>;
  static_assert(TN == 1 || TN % 2 == 0, "columns of a thread come in adjacent pairs");
  constexpr int WX = T::TX < 4 ? T::TX : 4, WY = 32 / WX;  // threads of a warp
  static_assert(T::NG % 32 == 0 && T::TY % WY == 0, "whole warps per product");
  // A in pairs of rows where a thread has several: rows 2 ty, 2 ty + 1, ...
  __shared__ __align__(16) float2 As[2][NB][BK][BM + 2];
  __shared__ __align__(16) float2 Bs[2][NB][BK][BN + 2];
  const int g = NB > 1 ? threadIdx.x / T::NG : 0;   // product of the block
  const int tid = NB > 1 ? threadIdx.x % T::NG : threadIdx.x;
  const int w = tid / 32, l = tid % 32;
  const int tx = (w % (T::TX / WX)) * WX + l % WX, ty = (w / (T::TX / WX)) * WY + l / WX;
  const int64_t tile = (int64_t)blockIdx.x * NB + g;
  const int64_t z = tile / (mt * nt);
  const int64_t rem = tile - z * (mt * nt);
  const int64_t m0 = rem / nt * BM, n0 = rem % nt * BN;
  const bool live = z < batch;
  // this thread's chunks: row r, k pair c of the tile
  const float2 *pa[T::PA], *pb[T::PB];
  bool oka[T::PA], okb[T::PB];
#pragma unroll
  for (int i = 0; i < T::PA; i++) {
    const int ch = tid + i * T::NG, r = ch / (BK / 2), c = ch % (BK / 2);
    oka[i] = live && ch < T::CA && m0 + r < M;
    pa[i] = A + (oka[i] ? z * sA + (m0 + r) * K + 2 * c : 0);
  }
#pragma unroll
  for (int i = 0; i < T::PB; i++) {
    const int ch = tid + i * T::NG, r = ch / (BK / 2), c = ch % (BK / 2);
    okb[i] = live && ch < T::CB && n0 + r < N;
    pb[i] = B + (okb[i] ? z * sB + (n0 + r) * K + 2 * c : 0);
  }
  const int kc = 2 * (tid % (BK / 2));  // k of this thread's chunks within a tile
  static_assert(T::NG % (BK / 2) == 0, "a thread's chunks share their k pair");
  float4 ra[T::PA], rb[T::PB];
  auto load = [&](int64_t k0) {
    auto get = [&](const float2 *p, bool ok) {
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (vec) {
        if (ok && k0 + kc < K) v = *reinterpret_cast<const float4 *>(p + k0);
      } else {
        if (ok && k0 + kc < K) v.x = p[k0].x, v.y = p[k0].y;
        if (ok && k0 + kc + 1 < K) v.z = p[k0 + 1].x, v.w = p[k0 + 1].y;
      }
      return v;
    };
#pragma unroll
    for (int i = 0; i < T::PA; i++) ra[i] = get(pa[i], oka[i]);
#pragma unroll
    for (int i = 0; i < T::PB; i++) rb[i] = get(pb[i], okb[i]);
  };
  auto store = [&](int s) {
#pragma unroll
    for (int i = 0; i < T::PA; i++) {
      const int ch = tid + i * T::NG, r = ch / (BK / 2);
      if (T::CA % T::NG == 0 || ch < T::CA) {
        As[s][g][kc][r] = make_float2(ra[i].x, ra[i].y);
        As[s][g][kc + 1][r] = make_float2(ra[i].z, ra[i].w);
      }
    }
#pragma unroll
    for (int i = 0; i < T::PB; i++) {
      const int ch = tid + i * T::NG, r = ch / (BK / 2);
      if (T::CB % T::NG == 0 || ch < T::CB) {
        Bs[s][g][kc][r] = make_float2(rb[i].x, rb[i].y);
        Bs[s][g][kc + 1][r] = make_float2(rb[i].z, rb[i].w);
      }
    }
  };
  // columns of this thread: pairs 2 tx, 2 tx + 1, then 2 TX further on
  auto col = [&](int j) { return TN == 1 ? tx : 2 * tx + (j & 1) + (j >> 1) * 2 * T::TX; };
  auto row = [&](int i) { return 2 * ty + (i & 1) + (i >> 1) * 2 * T::TY; };
  float2 acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; i++)
#pragma unroll
    for (int j = 0; j < TN; j++) acc[i][j] = make_float2(0.f, 0.f);
  load(0);
  store(0);
  __syncthreads();
  int s = 0;
  for (int64_t k0 = 0; k0 < K; k0 += BK, s ^= 1) {
    const bool more = k0 + BK < K;
    if (more) load(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; kk++) {
      float2 a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; i += 2) {
        const float4 v = *reinterpret_cast<const float4 *>(&As[s][g][kk][row(i)]);
        a[i] = make_float2(v.x, v.y);
        a[i + 1] = make_float2(v.z, v.w);
      }
      if (TN == 1) {
        b[0] = Bs[s][g][kk][tx];
      } else {
#pragma unroll
        for (int j = 0; j < TN; j += 2) {
          const float4 v = *reinterpret_cast<const float4 *>(&Bs[s][g][kk][col(j)]);
          b[j] = make_float2(v.x, v.y);
          b[j + (TN > 1)] = make_float2(v.z, v.w);
        }
      }
#pragma unroll
      for (int i = 0; i < TM; i++)
#pragma unroll
        for (int j = 0; j < TN; j++) {
          acc[i][j].x = fmaf(a[i].x, b[j].x, acc[i][j].x);
          acc[i][j].y = fmaf(a[i].x, b[j].y, acc[i][j].y);
        }
#pragma unroll
      for (int i = 0; i < TM; i++)
#pragma unroll
        for (int j = 0; j < TN; j++) {
          acc[i][j].x = fmaf(-a[i].y, b[j].y, acc[i][j].x);
          acc[i][j].y = fmaf(a[i].y, b[j].x, acc[i][j].y);
        }
    }
    if (more) {
      store(s ^ 1);
      __syncthreads();
    }
  }
  if (!live) return;
  if (!scatter) {
    float2 *Cz = C + z * sC;
    const bool pair = TN > 1 && (N & 1) == 0 && ((sC & 1) == 0) && (reinterpret_cast<uintptr_t>(C) & 15) == 0;
#pragma unroll
    for (int i = 0; i < TM; i++) {
      const int64_t m = m0 + row(i);
      if (m >= M) continue;
#pragma unroll
      for (int j = 0; j < TN; j += 2) {
        const int64_t n = n0 + col(j);
        if (pair) {
          if (n < N) {
            const float2 u = acc[i][j], v = acc[i][j + (TN > 1)];
            *reinterpret_cast<float4 *>(Cz + m * N + n) = make_float4(u.x, u.y, v.x, v.y);
          }
        } else {
          if (n < N) Cz[m * N + n] = acc[i][j];
          if (TN > 1 && n + 1 < N) Cz[m * N + n + 1] = acc[i][j + (TN > 1)];
        }
      }
    }
  } else {
    const int64_t ob = scatter_bits(z, sc.nb, sc.pb);
    int64_t on[TN];
#pragma unroll
    for (int j = 0; j < TN; j++) on[j] = scatter_bits(n0 + col(j), sc.nn, sc.pn);
#pragma unroll
    for (int i = 0; i < TM; i++) {
      const int64_t m = m0 + row(i);
      if (m >= M) continue;
      const int64_t om = ob + scatter_bits(m, sc.nm, sc.pm);
#pragma unroll
      for (int j = 0; j < TN; j++)
        if (n0 + col(j) < N) C[om + on[j]] = acc[i][j];
    }
  }
}

template <int BM, int BN, int TM, int TN, int BK, int NB, int MINB>
cudaError_t run_tile(const float2 *A, const float2 *B, float2 *C, int64_t batch, int64_t M, int64_t N, int64_t K,
                     int64_t sA, int64_t sB, int64_t sC, const CScatter *sc, cudaStream_t s) {
  const int64_t mt = (M + BM - 1) / BM, nt = (N + BN - 1) / BN;
  const int vec = (K % 2) == 0 && (sA % 2) == 0 && (sB % 2) == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0 &&
                  (reinterpret_cast<uintptr_t>(B) & 15) == 0;
  CScatter none{};
  // A grid has at most 2^31 - 1 blocks: a batch of more tiles (of operands
  // with strides of zero, say) goes in parts of 2^j products. (The first tile
  // as a kernel argument cost every launch up to 6 %.)
  int64_t part = batch;
  if ((mt * nt * batch + NB - 1) / NB > 0x7fffffff) {
    if (mt * nt > 0x7fffffff) return cudaErrorInvalidValue;
    for (part = 1; 2 * part * mt * nt <= 0x7fffffff;) part *= 2;
  }
  for (int64_t z0 = 0; z0 < batch; z0 += part) {
    const int64_t n = std::min(part, batch - z0);
    cgemm_tile_kernel<BM, BN, TM, TN, BK, NB, MINB>
        <<<(unsigned)((mt * nt * n + NB - 1) / NB), TileCfg<BM, BN, TM, TN, BK, NB>::NT, 0, s>>>(
            A + z0 * sA, B + z0 * sB, C + (sc ? scatter_bits(z0, sc->nb, sc->pb) : z0 * sC), n, M, N, K, sA, sB, sC,
            sc ? *sc : none, sc ? 1 : 0, vec, mt, nt);
  }
  return cudaGetLastError();
}

// Which tile: the largest whose blocks still fill the chip, then smaller ones.
// Measured, before (64 x 64 tiles of 4 x 4, 128 x 16 and 256 x 4) -> after:
//   b16 M2048 N256 K256 446 -> 308 us (56 TF/s of 80 FP32), M4096 N2048 K1024
//   1626 -> 1200; b32768 M32 N8 K64 1589 -> 152 us (4.9 TB/s);
//   b2048 M64 N4 K64 58 -> 19; b5 M1000 N77 K123 38 -> 19 (64 x 64 tiles,
//   160 blocks: 31); b8 M256 N64 K64 17 -> 7; b1 M128 N128 K128 31 -> 7.
cudaError_t launch_tiled(const float2 *A, const float2 *B, float2 *C, int64_t batch, int64_t M, int64_t N, int64_t K,
                         int64_t sA, int64_t sB, int64_t sC, const CScatter *sc, cudaStream_t s) {
  auto blocks = [&](int bm, int bn) { return ((M + bm - 1) / bm) * ((N + bn - 1) / bn) * batch; };
  if (N <= 4 && K > 8) return run_tile<64, 4, 4, 1, 16, 2, 4>(A, B, C, batch, M, N, K, sA, sB, sC, sc, s);
  // few columns and a short sum (below 256 rows, where the skinny kernels start):
  // bound by a tile's start and end, so no padded columns and a K tile of four
  // (64 x 16 -> 64 x 4 tiles: b4096 M255 N2 K4 45 -> 16 us, b4096 M96 N1 K1 25 ->
  // 10, b20000 M128 N2 K8 117 -> 62, 60 with a K tile of eight)
  if (N <= 4 && M >= 64) return run_tile<64, 4, 4, 1, 4, 2, 4>(A, B, C, batch, M, N, K, sA, sB, sC, sc, s);
  if (N <= 16) {
    // few summed values: a short K tile, more rows a block
    if (K <= 8 && M >= 64) return run_tile<64, 16, 4, 2, 8, 2, 3>(A, B, C, batch, M, N, K, sA, sB, sC, sc, s);
    if (N <= 8)
      return M > 16 ? run_tile<32, 8, 2, 2, 16, 2, 4>(A, B, C, batch, M, N, K, sA, sB, sC, sc, s)
                    : run_tile<16, 8, 2, 1, 16, 4, 2>(A, B, C, batch, M, N, K, sA, sB, sC, sc, s);
    if (M > 16 && blocks(32, 16) >= 152) return run_tile<32, 16, 4, 2, 16, 2, 4>(A, B, C, batch, M, N, K, sA, sB, sC, sc, s);
    return run_tile<16, 16, 2, 2, 16, 2, 3>(A, B, C, batch, M, N, K, sA, sB, sC, sc, s);
  }
  if (N > 32 && M > 32 && blocks(64, 64) >= 2 * 152)
    return run_tile<64, 64, 8, 4, 8, 1, 3>(A, B, C, batch, M, N, K, sA, sB, sC, sc, s);
  if (M > 32 && blocks(64, 32) >= 200) return run_tile<64, 32, 4, 4, 8, 1, 4>(A, B, C, batch, M, N, K, sA, sB, sC, sc, s);
  if (blocks(32, 32) >= 100) return run_tile<32, 32, 4, 2, 8, 1, 4>(A, B, C, batch, M, N, K, sA, sB, sC, sc, s);
  return run_tile<16, 16, 2, 2, 16, 2, 3>(A, B, C, batch, M, N, K, sA, sB, sC, sc, s);
}
