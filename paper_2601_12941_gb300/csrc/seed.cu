// Integer-pixel seed search: for every seed, the ZNCC between the reference subset
// and the deformed subset shifted by each integer offset (du, dv), |du|, |dv| <= R,
// whose pixels all lie inside the deformed image. Integer gray levels are summed
// exactly in 64-bit integers and normalised once in FP64:
//     C = (N Sfg - Sf Sg) / sqrt((N Sff - Sf^2) (N Sgg - Sg^2)),
// so ranking ties are decided on exact values. The best offset (larger C, then
// smaller |du|+|dv|, then smaller dv, then smaller du) starts the seed's IC-GN
// (Sec. 2.2 leaves the initial estimate to an FFT stage; a brute-force integer
// search gives the same integer start for a seed).
#include <math.h>

#include "dic_internal.cuh"

namespace dic {
namespace {

constexpr double kNoScore = -2.0;    // offset not usable (out of the image or flat)
constexpr double kFlatRef = -3.0;    // the reference subset itself is flat

__device__ __forceinline__ bool integer_gray(int dtype) { return dtype == DIC_U8 || dtype == DIC_U16; }

// sum over the G lanes (a power of two) that share an offset
template <int G, typename V>
__device__ __forceinline__ V seed_sum(V v) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// gray level of a pixel as the sums take it: an exact integer, or FP64
template <typename V>
__device__ __forceinline__ V seed_gray(const GrayPlane& g, int64_t x, int64_t y) {
  if constexpr (sizeof(V) == sizeof(int32_t))
    return static_cast<V>(load_gray<float>(g, x, y));
  else
    return load_gray<double>(g, x, y);
}

// The scores of one row of offsets: F holds the gray levels (int32 or FP64), A is the type
// of the sums (int64: exact, so their order does not matter, or FP64). The block stages the
// reference subset and, where shared memory holds them (staged), the S rows of the
// deformed image that the row of offsets covers; then G lanes per offset, over its pixels.
// Bound: the latency of one offset's pixels over G where there are few offsets, else the three
// additions per pixel, and the sums over the lanes where a lane has few pixels.
template <int G, typename F, typename A>
__device__ void seed_row_scores(const SeedArgs& a, F* f, bool staged, int xc, int yc, int dv, double* out) {
  const int S = a.S, r = (a.S - 1) / 2, N = S * S, SW = S + 2 * a.R;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  F* gs = f + N;                       // [S][SW]: columns xc - r - R ..., 0 outside the image
  for (int e = threadIdx.x; e < N; e += blockDim.x) f[e] = seed_gray<F>(a.ref, xc - r + e % S, yc - r + e / S);
  if (staged) {
#pragma unroll 4
    for (int e = threadIdx.x; e < S * SW; e += blockDim.x) {
      const int x = xc - r - a.R + e % SW, y = yc + dv - r + e / SW;
      gs[e] = x >= 0 && y >= 0 && x < a.W && y < a.H ? seed_gray<F>(a.def, x, y) : F(0);
    }
  }
  __syncthreads();
  A Sf = 0, Sff = 0;
  for (int e = lane; e < N; e += 32) {
    const A v = f[e];
    Sf += v;
    Sff += v * v;
  }
  Sf = seed_sum<32>(Sf);
  Sff = seed_sum<32>(Sff);
  const A Df = static_cast<A>(N) * Sff - Sf * Sf;
  constexpr int PW = 32 / G;           // offsets per warp
  const int part = lane & (G - 1);
  for (int d0 = warp * PW; d0 < 2 * a.R + 1; d0 += nw * PW) {
    const int du = d0 + lane / G - a.R;
    const int x0 = xc + du - r, y0 = yc + dv - r;
    const bool in = du <= a.R && x0 >= 0 && y0 >= 0 && x0 + S <= a.W && y0 + S <= a.H;
    double score = kNoScore;
    if (!(Df > 0)) {
      score = kFlatRef;
    } else if (__any_sync(0xffffffffu, in)) {   // (without the vote 28 instead of 15 us at subset 21, radius 8)
      A Sg = 0, Sgg = 0, Sfg = 0;
      if (in) {
        int xx = part % S, yy = part / S;
        for (int e = part; e < N; e += G) {
          const A g = staged ? gs[yy * SW + (du + a.R) + xx] : seed_gray<F>(a.def, x0 + xx, y0 + yy);
          Sg += g;
          Sgg += g * g;
          Sfg += g * static_cast<A>(f[e]);
          for (xx += G; xx >= S; xx -= S) ++yy;
        }
      }
      Sg = seed_sum<G>(Sg);
      Sgg = seed_sum<G>(Sgg);
      Sfg = seed_sum<G>(Sfg);
      const A Dg = static_cast<A>(N) * Sgg - Sg * Sg;
      if (in && Dg > 0) {
        const A num = static_cast<A>(N) * Sfg - Sf * Sg;
        score = sizeof(F) == sizeof(int32_t)
                    ? static_cast<double>(num) / sqrt(static_cast<double>(Df) * static_cast<double>(Dg))
                    : static_cast<double>(num) / sqrt(static_cast<double>(Df * Dg));
      }
    }
    if (part == 0 && du <= a.R) out[du + a.R] = score;
  }
}

// grid (2R+1, n_seeds): block y = seed, block x = dv + R; warps stride over du
template <int G>
__global__ void __launch_bounds__(256) seed_scores_kernel(SeedArgs a, int staged) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int s = blockIdx.y;
  const int dv = static_cast<int>(blockIdx.x) - a.R;
  const int xc = a.seed_xy[2 * s], yc = a.seed_xy[2 * s + 1];
  const int side = 2 * a.R + 1;
  double* out = a.scores + static_cast<int64_t>(s) * side * side + (dv + a.R) * side;
  if (integer_gray(a.ref.dtype) && integer_gray(a.def.dtype))
    seed_row_scores<G, int32_t, int64_t>(a, reinterpret_cast<int32_t*>(smem_raw), staged != 0, xc, yc, dv, out);
  else
    seed_row_scores<G, double, double>(a, reinterpret_cast<double*>(smem_raw), staged != 0, xc, yc, dv, out);
}

// one block per seed: the best offset (larger C, then smaller |du|+|dv|, then
// smaller dv, then smaller du) into best[s]; -1 if no offset is usable, -2 if the
// reference subset is flat
__global__ void __launch_bounds__(256) seed_best_kernel(SeedCommitArgs a) {
  const int s = blockIdx.x;
  const int side = 2 * a.R + 1;
  const double* sc = a.scores + static_cast<int64_t>(s) * side * side;
  double bc = 0.0;
  int bkey = 0x7fffffff, be = -1, flat = 0;
  for (int e = threadIdx.x; e < side * side; e += blockDim.x) {
    const double c = sc[e];
    if (c == kFlatRef) flat = 1;
    if (c < -1.5) continue;
    const int du = e % side - a.R, dv = e / side - a.R;
    const int key = ((abs(du) + abs(dv)) * (side + 1) + (dv + a.R)) * (side + 1) + (du + a.R);
    if (be < 0 || c > bc || (c == bc && key < bkey)) {
      be = e;
      bc = c;
      bkey = key;
    }
  }
  __shared__ double s_c[8];
  __shared__ int s_k[8], s_e[8], s_f[8];
  for (int o = 16; o > 0; o >>= 1) {
    const double oc = __shfl_xor_sync(0xffffffffu, bc, o);
    const int ok = __shfl_xor_sync(0xffffffffu, bkey, o);
    const int oe = __shfl_xor_sync(0xffffffffu, be, o);
    flat |= __shfl_xor_sync(0xffffffffu, flat, o);
    if (oe >= 0 && (be < 0 || oc > bc || (oc == bc && ok < bkey))) {
      bc = oc;
      bkey = ok;
      be = oe;
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) {
    s_c[warp] = bc;
    s_k[warp] = bkey;
    s_e[warp] = be;
    s_f[warp] = flat;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < static_cast<int>(blockDim.x / 32); ++w) {
      flat |= s_f[w];
      if (s_e[w] >= 0 && (be < 0 || s_c[w] > bc || (s_c[w] == bc && s_k[w] < bkey))) {
        bc = s_c[w];
        bkey = s_k[w];
        be = s_e[w];
      }
    }
    a.best[s] = be >= 0 ? be : (flat ? -2 : -1);
  }
}

// one thread: seeds in the order given, duplicates and out-of-ROI seeds skipped
__global__ void seed_commit_kernel(SeedCommitArgs a) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const int side = 2 * a.R + 1;
  int count = 0;
  for (int s = 0; s < a.n_seeds; ++s) {
    const int q = a.seed_q[s];
    if (a.roi_ok && !a.roi_ok[q]) continue;
    if (a.wave[q] >= 0) continue;
    a.wave[q] = 0;
    double* p = a.p + static_cast<int64_t>(q) * a.nparams;
    if (a.fft_u) {
      for (int c = 0; c < a.nparams; ++c) p[c] = 0.0;
      p[0] = floor(static_cast<double>(a.fft_u[q]) + 0.5);
      p[1] = floor(static_cast<double>(a.fft_v[q]) + 0.5);
      a.frontier0[count++] = q;
      continue;
    }
    const int best = a.best[s];
    if (best < 0) {
      a.status[q] = best == -2 ? DIC_PT_FLAT : DIC_PT_OUT_OF_BOUNDS;
      continue;
    }
    for (int c = 0; c < a.nparams; ++c) p[c] = 0.0;
    p[0] = static_cast<double>(best % side - a.R);
    p[1] = static_cast<double>(best / side - a.R);
    a.frontier0[count++] = q;
  }
  a.counters[kCount + 0] = count;
  a.counters[kCount + 1] = 0;
  a.counters[kCount + 2] = 0;
  a.counters[kWork + 0] = 0;
  a.counters[kWork + 1] = 0;
  a.counters[kWork + 2] = 0;
}

}  // namespace

cudaError_t launch_seed_scores(const SeedArgs& a, cudaStream_t s) {
  const bool exact = (a.ref.dtype == DIC_U8 || a.ref.dtype == DIC_U16) &&
                     (a.def.dtype == DIC_U8 || a.def.dtype == DIC_U16);
  const size_t es = exact ? sizeof(int32_t) : sizeof(double);
  size_t smem = es * a.S * a.S;
  const size_t rows = es * a.S * (a.S + 2 * static_cast<size_t>(a.R));
  const int staged = smem + rows <= 48 * 1024;   // (up to radius 39 at subset 61 for integer gray levels)
  if (staged) smem += rows;
  // Lanes per offset. A whole warp is fastest while the offsets are few, so that one's pixels are the
  // call (subset 21, radius 8: 15 us; 8 lanes 12, one lane 31), and at subsets of 51 and up, where its sums
  // over the lanes cost little at any radius. With more offsets than the SMs' warps they
  // cost more than a small subset's pixels (us with 32 / 8 / 2 / 1 lanes, u8, one seed, radius 256: subset
  // 5 364 / 100 / 35 / 24, 15 386 / 134 / 94 / 90, 21 389 / 193 / 164 / 162, 61 1821 / 1595 / 1500 / 1593; FP32 gray
  // levels at 61, radius 32: 371 / 440 / 493 / 884).
  const int64_t offsets = static_cast<int64_t>(2 * a.R + 1) * (2 * a.R + 1) * a.n_seeds;
  const int lanes = offsets <= 2048 ? (a.S >= 17 ? 32 : 8) : a.S >= 51 ? 32 : a.S >= 17 ? 8 : a.S >= 9 ? 2 : 1;
  dim3 grid(2 * a.R + 1, a.n_seeds);
  switch (lanes) {
    case 1: seed_scores_kernel<1><<<grid, 256, smem, s>>>(a, staged); break;
    case 2: seed_scores_kernel<2><<<grid, 256, smem, s>>>(a, staged); break;
    case 8: seed_scores_kernel<8><<<grid, 256, smem, s>>>(a, staged); break;
    default: seed_scores_kernel<32><<<grid, 256, smem, s>>>(a, staged);
  }
  return cudaGetLastError();
}

cudaError_t launch_seed_commit(const SeedCommitArgs& a, cudaStream_t s) {
  if (!a.fft_u) seed_best_kernel<<<a.n_seeds, 256, 0, s>>>(a);
  seed_commit_kernel<<<1, 32, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace dic
