// Strain post-processing (Sec. 2.3): at every grid point the displacement gradient
// of a least-squares fit u = P c over the N x N window of grid points centred on it
// (Eq. 8-9; P = [1, x, y] or [1, x, y, x^2, y^2, x^2 y, x y^2, x^2 y^2]), the
// deformation gradient F = I + grad u (Eq. 6) and one of the five strain measures.
//
// Only accepted points (status 0) inside the grid enter a window, and the centre
// must be accepted. A full window (every point present) is the common case: there
// the odd-in-x basis terms {x, x y^2} are orthogonal to the others, so the fitted
// x slope is sum_ij i (a + b j^2) u_ij / s in grid units (i, j) with two constants
// a, b of the window, and the y slope sum_ij j (a + b i^2) u_ij / s, applied
// separably from shared-memory tiles. A window with missing points is fitted
// from its normal equations (grid units, unit-diagonal scaling, elimination
// without exchanges); a scaled pivot at or below 1e-5 leaves the point without
// strain (NaN). Arithmetic in FP32 on displacement offsets: from a reference point of
// the tile for the separable filter (whose slope weights sum to zero, so the reference
// drops out), from the centre, rounded once, for the general fit.
#include <math.h>

#include "dic_internal.cuh"

namespace dic {
namespace {

constexpr float kMinScaledPivot = 1e-5f;

// P(x, y) for the basis (Eq. 9, as printed)
__device__ __forceinline__ void basis_row(int basis, float x, float y, float* P) {
  P[0] = 1.0f;
  P[1] = x;
  P[2] = y;
  if (basis != DIC_STRAIN_BILINEAR) {
    P[3] = x * x;
    P[4] = y * y;
    P[5] = x * x * y;
    P[6] = x * y * y;
    P[7] = x * x * y * y;
  }
}

// An FP64 number that is an FP32 number, zero or normal, as the mixed path writes them (the low
// 29 bits of the pattern zero, exponent 897 ... 1150): its FP32 bits on the integer pipe.
// False for any other.
__device__ __forceinline__ bool exact_float(double u, float* f) {
  const int hi = __double2hiint(u), lo = __double2loint(u);
  const int e = (hi >> 20) & 0x7ff;
  const bool zero = ((hi & 0x7fffffff) | lo) == 0;
  const int bits = zero ? 0 : (((e - 896) << 23) | ((hi & 0xfffff) << 3) | static_cast<int>(static_cast<unsigned>(lo) >> 29));
  *f = __int_as_float((hi & 0x80000000) | bits);
  return zero || ((lo & 0x1fffffff) == 0 && e > 896 && e < 1151);
}
// u rounded to FP32 (the FP64 pipe, which converts, runs at 1/64 of the FP32 rate here)
__device__ __forceinline__ float to_float(double u) {
  float f;
  // (volatile: not hoisted above the test)
  if (!exact_float(u, &f)) asm volatile("cvt.rn.f32.f64 %0, %1;" : "=f"(f) : "d"(u));
  return f;
}
// u - uc rounded once to FP32: of two FP32 numbers (uc32: uc = ucf is one) one FP32 subtraction
// rounds the same exact difference, otherwise it is formed in FP64.
__device__ __forceinline__ float offset_from(double u, double uc, float ucf, bool uc32) {
  float f;
  if (uc32 && exact_float(u, &f)) return f - ucf;
  return static_cast<float>(u - uc);
}

// General least squares over the valid points of the window (out of line: windows with
// missing points are the rare case) for a basis of K terms: returns NaN in .x when the
// design is not well posed; else the x and y slopes (grid units) of u and v. Which
// points are present comes from the block's staged values su (row pitch SX; NaN where
// a point is missing or outside the grid; centre at slot ec); the displacements are read
// again as FP64 (q: the centre's grid point) and their offsets from the centre rounded
// once. Normal equations with
// unit-diagonal scaling, then elimination without exchanges, indexed at compile time
// (K fixed) so that the matrix lives in registers.
template <int K>
__device__ __noinline__ float4 fit_window(const StrainArgs& a, int h, const float* su, int SX, int ec, int64_t q) {
  const float4 fail = make_float4(__int_as_float(0x7fc00000), 0.0f, 0.0f, 0.0f);
  const double uc = a.u[q], vc = a.v[q];
  float ucf, vcf;
  const bool uc32 = exact_float(uc, &ucf), vc32 = exact_float(vc, &vcf);
  float M[K][K], ru[K], rv[K];
#pragma unroll
  for (int r = 0; r < K; ++r) {
    ru[r] = rv[r] = 0.0f;
#pragma unroll
    for (int c = 0; c < K; ++c) M[r][c] = 0.0f;
  }
  int count = 0;
  for (int dj = -h; dj <= h; ++dj) {
    for (int di = -h; di <= h; ++di) {
      const int e = ec + dj * SX + di;
      if (su[e] != su[e]) continue;                  // missing: not accepted, or outside the grid
      float P[8];
      basis_row(a.basis, static_cast<float>(di), static_cast<float>(dj), P);
      const int64_t qe = q + static_cast<int64_t>(dj) * a.nx + di;
      const float du = offset_from(a.u[qe], uc, ucf, uc32), dv = offset_from(a.v[qe], vc, vcf, vc32);
#pragma unroll
      for (int r = 0; r < K; ++r) {
        ru[r] += P[r] * du;
        rv[r] += P[r] * dv;
#pragma unroll
        for (int c = r; c < K; ++c) M[r][c] += P[r] * P[c];
      }
      ++count;
    }
  }
  if (count < K) return fail;
  float d[K];
#pragma unroll
  for (int r = 0; r < K; ++r) {
    if (!(M[r][r] > 0.0f)) return fail;
    d[r] = rsqrtf(M[r][r]);
  }
#pragma unroll
  for (int r = 0; r < K; ++r) {
#pragma unroll
    for (int c = r; c < K; ++c) M[r][c] *= d[r] * d[c];
#pragma unroll
    for (int c = 0; c < r; ++c) M[r][c] = M[c][r];
    ru[r] *= d[r];
    rv[r] *= d[r];
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const float piv = M[k][k];
    if (!(piv > kMinScaledPivot)) return fail;
    const float inv = 1.0f / piv;
#pragma unroll
    for (int r = k + 1; r < K; ++r) {
      const float f = M[r][k] * inv;
#pragma unroll
      for (int c = k + 1; c < K; ++c) M[r][c] -= f * M[k][c];
      ru[r] -= f * ru[k];
      rv[r] -= f * rv[k];
    }
  }
#pragma unroll
  for (int r = K - 1; r >= 0; --r) {
    float xu = ru[r], xv = rv[r];
#pragma unroll
    for (int c = r + 1; c < K; ++c) {
      xu -= M[r][c] * ru[c];
      xv -= M[r][c] * rv[c];
    }
    ru[r] = xu / M[r][r];
    rv[r] = xv / M[r][r];
  }
  // undo the scaling: coefficient r is d[r] z[r]
  return make_float4(d[1] * ru[1], d[2] * ru[2], d[1] * rv[1], d[2] * rv[2]);
}

// eigenvalues mu1 >= mu2 of the symmetric [[d11, d12], [d12, d22]]
__device__ __forceinline__ void sym_eig(float d11, float d12, float d22, float* mu1, float* mu2) {
  const float m = 0.5f * (d11 + d22);
  const float q = sqrtf(0.25f * (d11 - d22) * (d11 - d22) + d12 * d12);
  *mu1 = m + q;
  *mu2 = m - q;
}

// f(I + D) = m I + g (D - tr(D)/2 I) for a symmetric D with eigenvalues mu1, mu2,
// where m is the mean of f at 1 + mu_k and g their divided difference
__device__ __forceinline__ void spectral(float d11, float d12, float d22, float m, float g, float* e) {
  const float t = 0.5f * (d11 + d22);
  e[0] = m + g * (d11 - t);
  e[1] = m + g * (d22 - t);
  e[2] = g * d12;
}

// Sec. 2.3: strain (exx, eyy, exy) from H = grad u, formed from the small parts of
// F^T F = I + D or F F^T = I + D' so that no 1 is subtracted from a near-1 value.
__device__ __forceinline__ void strain_from_gradient(int measure, float h11, float h12, float h21, float h22,
                                                     float* e) {
  const bool left = measure == DIC_EULER_ALMANSI || measure == DIC_BIOT_LEFT;
  // D = H + H^T + H^T H (right) or D' = H + H^T + H H^T (left)
  const float d11 = left ? 2.0f * h11 + h11 * h11 + h12 * h12 : 2.0f * h11 + h11 * h11 + h21 * h21;
  const float d22 = left ? 2.0f * h22 + h21 * h21 + h22 * h22 : 2.0f * h22 + h12 * h12 + h22 * h22;
  const float d12 = left ? h12 + h21 + h11 * h21 + h12 * h22 : h12 + h21 + h11 * h12 + h21 * h22;
  if (measure == DIC_GREEN_LAGRANGE) {            // (F^T F - I) / 2
    e[0] = 0.5f * d11;
    e[1] = 0.5f * d22;
    e[2] = 0.5f * d12;
    return;
  }
  if (measure == DIC_EULER_ALMANSI) {             // (I - (F F^T)^-1) / 2 = (D' + det D' I) / (2 det(I + D'))
    const float det = d11 * d22 - d12 * d12;
    const float s = 0.5f / (1.0f + d11 + d22 + det);
    e[0] = (d11 + det) * s;
    e[1] = (d22 + det) * s;
    e[2] = d12 * s;
    return;
  }
  float mu1, mu2;
  sym_eig(d11, d12, d22, &mu1, &mu2);
  if (measure == DIC_HENCKY) {                    // ln sqrt(C): f(lambda) = ln(lambda) / 2
    const float m = 0.25f * (log1pf(mu1) + log1pf(mu2));
    const float z = (mu1 - mu2) / (1.0f + mu2);
    const float l = z < 1e-3f ? 1.0f - z * (0.5f - z * (1.0f / 3.0f)) : log1pf(z) / z;
    spectral(d11, d12, d22, m, 0.5f * l / (1.0f + mu2), e);
    return;
  }
  // Biot, right or left: sqrt(I + D) - I: f(lambda) = sqrt(lambda) - 1
  const float r1 = sqrtf(1.0f + mu1), r2 = sqrtf(1.0f + mu2);
  const float m = 0.5f * (mu1 / (1.0f + r1) + mu2 / (1.0f + r2));
  spectral(d11, d12, d22, m, 1.0f / (r1 + r2), e);
}

constexpr int kTile = 32;         // grid points per block along x
constexpr int kStrainThreads = 256;    // threads per block
constexpr int kRun = 4;           // outputs per thread along x in the row sums
constexpr int kStrainWarps = kStrainThreads / 32;
constexpr int kStrainBlocksPerSm = 3;

// row pitch of the staged values: at least SX and 1 mod 4, so that the row pass (8 threads
// four columns apart in each of four rows) meets 32 distinct banks
__host__ __device__ constexpr int staged_pitch(int SX) { return SX + ((1 - SX) & 3); }

// Block of kTile x 8 R grid points, half-window H, R points per thread. The block stages the FP32 displacements of
// its points and of a halo of H points (NaN where a point is outside the grid or not
// accepted), then applies the full-window slope filter separably to offsets from one
// accepted point of the tile: along each staged row the sums
// fx = sum_i i d and g = a sum_i d + b sum_i i^2 d over the window's columns, then down each
// column the x slope sum_j (a + b j^2) fx_j and the y slope sum_j j g_j. Samples at -i and
// i enter as their sum and difference; a thread forms kRun (along x) or R (along y) neighbouring
// outputs from one set of loads. Each row's fx takes its middle sample with weight zero, so that a
// missing or infinite value anywhere in a window makes the x slope NaN or infinite (without
// it the centre column would reach only the y slope, and the point itself neither). Accepted
// points with such a window are collected and then share the block's threads for their general
// fits, so that a fit does not hold up a warp of 31 finished points. Bound: HBM (46 bytes a
// point) and latency. 10.7 M points, window 9, biquadratic, Green-Lagrange, a band and stray
// points rejected: 336 us (743 us with one output per thread and fits where they fell; 458 us at four
// blocks per SM, whose 64 registers spill the fits).
template <int H, int R>
__global__ void __launch_bounds__(kStrainThreads, kStrainBlocksPerSm) strain_kernel(const __grid_constant__ StrainArgs a) {
  constexpr int TY = R * kStrainWarps;
  constexpr int N = 2 * H + 1, SX = kTile + 2 * H, SY = TY + 2 * H, PX = staged_pitch(SX);
  constexpr int kRows = (SY + kStrainWarps - 1) / kStrainWarps;      // staged rows per warp
  extern __shared__ __align__(16) float smf[];
  float* rows = smf;                          // [4][SY][kTile] row sums: fx of u, g of u, fx of v, g of v
  float* su = rows + 4 * SY * kTile;          // [SY][PX] staged u
  float* sv = su + SY * PX;                   // ... v
  __shared__ float3 s_ref[kStrainWarps];           // first accepted finite point of each warp's tile rows: place (or 1e9), u, v
  __shared__ int s_fits;                      // points left to the general fit
  __shared__ short s_list[kTile * TY];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int x0 = blockIdx.x * kTile, y0 = blockIdx.y * TY;
  const float nan_ = __int_as_float(0x7fc00000);
  if (tid == 0) s_fits = 0;

  // ---- stage: warp w takes rows w, w + 8, ...; two columns per lane (the second in the halo)
  {
    double u[kRows][2], v[kRows][2];
    uint8_t st[kRows][2];
#pragma unroll
    for (int k = 0; k < kRows; ++k)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int row = warp + k * kStrainWarps, col = lane + 32 * c;
        const int i = x0 - H + col, j = y0 - H + row;
        st[k][c] = 1;
        u[k][c] = v[k][c] = 0.0;
        if (row < SY && col < SX && i >= 0 && i < a.nx && j >= 0 && j < a.ny) {
          const int64_t q = static_cast<int64_t>(j) * a.nx + i;
          st[k][c] = a.status[q];
          u[k][c] = a.u[q];
          v[k][c] = a.v[q];
        }
      }
    float first = 1e9f, ru = 0.0f, rv = 0.0f;
#pragma unroll
    for (int k = 0; k < kRows; ++k)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int row = warp + k * kStrainWarps, col = lane + 32 * c;
        const bool ok = st[k][c] == 0;
        const float fu = to_float(u[k][c]), fv = to_float(v[k][c]);
        if (row < SY && col < SX) {
          su[row * PX + col] = ok ? fu : nan_;
          sv[row * PX + col] = ok ? fv : nan_;
        }
        // (a point of the tile itself: the offsets of its own points stay small and exact whatever lies
        // in the halo)
        const bool own = c == 0 ? lane >= H : lane < H;
        const unsigned m = row >= H && row < H + TY ? __ballot_sync(0xffffffffu, ok && own && isfinite(fu) && isfinite(fv)) : 0u;
        if (m && first == 1e9f) {              // (the same on every lane)
          const int l = __ffs(m) - 1;
          first = static_cast<float>(row * SX + l + 32 * c);
          ru = __shfl_sync(0xffffffffu, fu, l);
          rv = __shfl_sync(0xffffffffu, fv, l);
        }
      }
    if (lane == 0) s_ref[warp] = make_float3(first, ru, rv);
  }
  __syncthreads();
  float3 ref = s_ref[0];
#pragma unroll
  for (int w = 1; w < kStrainWarps; ++w)
    if (s_ref[w].x < ref.x) ref = s_ref[w];

  // ---- row sums
  constexpr int kItems = SY * (kTile / kRun);
  for (int it = tid; it < 2 * kItems; it += kStrainThreads) {
    const int comp = it >= kItems ? 1 : 0, e = it - comp * kItems;
    const int row = e / (kTile / kRun), c0 = (e % (kTile / kRun)) * kRun;
    const float* src = (comp ? sv : su) + row * PX + c0;
    const float base = comp ? ref.z : ref.y;
    float d[N + kRun - 1];
#pragma unroll
    for (int k = 0; k < N + kRun - 1; ++k) d[k] = src[k] - base;
    float fx[kRun], g[kRun];
#pragma unroll
    for (int o = 0; o < kRun; ++o) {
      float sx = 0.0f * d[o + H], s0 = d[o + H], s2 = 0.0f;   // (zero, or NaN)
#pragma unroll
      for (int k = 1; k <= H; ++k) {
        const float p = d[o + H + k] + d[o + H - k], m = d[o + H + k] - d[o + H - k];
        sx = fmaf(static_cast<float>(k), m, sx);
        s0 += p;
        s2 = fmaf(static_cast<float>(k * k), p, s2);
      }
      fx[o] = sx;
      g[o] = fmaf(a.wa, s0, a.wb * s2);
    }
    float* dst = rows + (2 * comp * SY + row) * kTile + c0;
    *reinterpret_cast<float4*>(dst) = make_float4(fx[0], fx[1], fx[2], fx[3]);
    *reinterpret_cast<float4*>(dst + SY * kTile) = make_float4(g[0], g[1], g[2], g[3]);
  }
  __syncthreads();

  // ---- slopes: thread (column lane, rows R warp ..)
  const float inv_s = 1.0f / static_cast<float>(a.step);   // grid units -> pixels
  auto store = [&](int64_t q, bool ok, float4 gr) {
    if (ok) {
      const float h11 = gr.x * inv_s, h12 = gr.y * inv_s, h21 = gr.z * inv_s, h22 = gr.w * inv_s;
      float e[3];
      strain_from_gradient(a.measure, h11, h12, h21, h22, e);
      a.dudx[q] = h11;
      a.dudy[q] = h12;
      a.dvdx[q] = h21;
      a.dvdy[q] = h22;
      a.exx[q] = e[0];
      a.eyy[q] = e[1];
      a.exy[q] = e[2];
    } else {
      a.dudx[q] = a.dudy[q] = a.dvdx[q] = a.dvdy[q] = nan_;
      a.exx[q] = a.eyy[q] = a.exy[q] = nan_;
    }
    a.valid[q] = ok ? 1 : 0;
  };
  {
    const int r0 = warp * R;
    float gx[2][R], gy[2][R];
#pragma unroll
    for (int comp = 0; comp < 2; ++comp) {
      const float* f = rows + (2 * comp * SY + r0) * kTile + lane;
      float d[N + R - 1];
#pragma unroll
      for (int k = 0; k < N + R - 1; ++k) d[k] = f[k * kTile];
#pragma unroll
      for (int o = 0; o < R; ++o) {
        float s = a.wa * d[o + H];
#pragma unroll
        for (int k = 1; k <= H; ++k)
          s = fmaf(fmaf(a.wb, static_cast<float>(k * k), a.wa), d[o + H + k] + d[o + H - k], s);
        gx[comp][o] = s;
      }
#pragma unroll
      for (int k = 0; k < N + R - 1; ++k) d[k] = f[(SY + k) * kTile];
#pragma unroll
      for (int o = 0; o < R; ++o) {
        float s = 0.0f;
#pragma unroll
        for (int k = 1; k <= H; ++k) s = fmaf(static_cast<float>(k), d[o + H + k] - d[o + H - k], s);
        gy[comp][o] = s;
      }
    }
#pragma unroll
    for (int o = 0; o < R; ++o) {
      const int ic = x0 + lane, jc = y0 + r0 + o;
      if (ic >= a.nx || jc >= a.ny) continue;
      const int ec = (r0 + o + H) * PX + lane + H;
      const bool centre = su[ec] == su[ec];    // accepted (with u NaN: no strain either way)
      const bool full = isfinite(gx[0][o]) && isfinite(gy[0][o]) && isfinite(gx[1][o]) && isfinite(gy[1][o]);
      if (centre && !full)
        s_list[atomicAdd(&s_fits, 1)] = static_cast<short>((r0 + o) * kTile + lane);
      else
        store(static_cast<int64_t>(jc) * a.nx + ic, centre, make_float4(gx[0][o], gy[0][o], gx[1][o], gy[1][o]));
    }
  }
  __syncthreads();

  // ---- general fits, one thread each
  const int fits = s_fits;
  for (int k = tid; k < fits; k += kStrainThreads) {
    const int e = s_list[k], row = e / kTile, col = e % kTile;
    const int64_t q = static_cast<int64_t>(y0 + row) * a.nx + x0 + col;
    const int ec = (row + H) * PX + col + H;
    const float4 g = a.basis == DIC_STRAIN_BILINEAR ? fit_window<3>(a, H, su, PX, ec, q) : fit_window<8>(a, H, su, PX, ec, q);
    store(q, g.x == g.x, g);
  }
}

template <int H, int R>
cudaError_t launch_strain_rows(const StrainArgs& a, cudaStream_t s) {
  constexpr int TY = R * kStrainWarps, SX = kTile + 2 * H, SY = TY + 2 * H;
  constexpr int smem = static_cast<int>(sizeof(float)) * (4 * SY * kTile + 2 * SY * staged_pitch(SX));
  if (smem > 40 * 1024) {   // (thread-safe, once)
    static const cudaError_t configured =
        cudaFuncSetAttribute(strain_kernel<H, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (configured != cudaSuccess) return configured;
  }
  const dim3 grid((a.nx + kTile - 1) / kTile, (a.ny + TY - 1) / TY);
  strain_kernel<H, R><<<grid, kStrainThreads, smem, s>>>(a);
  return cudaGetLastError();
}

// Points per thread. Four share the halo best (3273 x 3273, window 9: 241 us, now 236; with two 278, with
// one 354). But a block whose points all need general fits runs R of them per thread, one after the
// other, and the call lasts as long as the turns of its blocks on the SMs. Small grids (a block's
// chain is the call: 100 x 70, window 21, every point accepted: 393 / 259 / 141 us with four / two /
// one) and grids whose last turn is nearly empty (1024 x 1024, FP64 displacements, 1 % missing, window
// 21: 4111 / 3666 / 3445 us) take fewer. Windows up to 9: where that saves an eighth of R x turns (at
// window 3, whose fits cost no more than the halo: where one turn does). From window 11 the border, all
// general fits, is a large part: one or two points up to ten turns, two from window 27 (1024 x
// 1024, window 21: 466 / 357 / 274 us; 3273 x 3273, window 31: 2136 / 1860 / 2264), two where one
// saves no turn (400 x 300, FP64, 1 % missing, window 21: 706 / 539 / 692).
template <int H>
cudaError_t launch_strain_half(const StrainArgs& a, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int64_t slots = static_cast<int64_t>(kStrainBlocksPerSm) * sms;
  auto turns = [&](int r) {
    const int64_t blocks = static_cast<int64_t>((a.nx + kTile - 1) / kTile) * ((a.ny + r * kStrainWarps - 1) / (r * kStrainWarps));
    return (blocks + slots - 1) / slots;
  };
  const int64_t t1 = turns(1), t2 = turns(2), t4 = turns(4);
  if constexpr (H == 1) {
    return t1 == 1 ? launch_strain_rows<H, 1>(a, s) : launch_strain_rows<H, 4>(a, s);
  } else {
    int r = 4;
    if (H <= 4) {
      if (8 * 2 * t2 <= 7 * 4 * t4) r = 2;
      if (8 * t1 <= 7 * r * (r == 2 ? t2 : t4)) r = 1;
    } else {
      r = t1 <= 10 && t1 < 2 * t2 ? 1 : t2 <= 10 || H > 12 ? 2 : 4;
    }
    if (r == 1) return launch_strain_rows<H, 1>(a, s);
    if (r == 2) return launch_strain_rows<H, 2>(a, s);
    if constexpr (H <= 12) return launch_strain_rows<H, 4>(a, s);
    return cudaErrorInvalidValue;   // (not reached: r <= 2 above window 25)
  }
}

}  // namespace

// one kernel per half-window (windows 3 ... 31), so that its sums are straight-line code
cudaError_t launch_strain(const StrainArgs& a, cudaStream_t s) {
  switch ((a.window - 1) / 2) {
    case 1: return launch_strain_half<1>(a, s);
    case 2: return launch_strain_half<2>(a, s);
    case 3: return launch_strain_half<3>(a, s);
    case 4: return launch_strain_half<4>(a, s);
    case 5: return launch_strain_half<5>(a, s);
    case 6: return launch_strain_half<6>(a, s);
    case 7: return launch_strain_half<7>(a, s);
    case 8: return launch_strain_half<8>(a, s);
    case 9: return launch_strain_half<9>(a, s);
    case 10: return launch_strain_half<10>(a, s);
    case 11: return launch_strain_half<11>(a, s);
    case 12: return launch_strain_half<12>(a, s);
    case 13: return launch_strain_half<13>(a, s);
    case 14: return launch_strain_half<14>(a, s);
    case 15: return launch_strain_half<15>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace dic
