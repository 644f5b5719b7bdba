// Model kernels of the XL-BOMD path: the Slater-Koster Hamiltonian H0, the
// periodic Ohno-Klopman Coulomb matrix gamma, H[n] = H0 + diag(gamma n), the
// Hellmann-Feynman forces (Eq. EqMotFT), Mulliken charges, and the
// velocity-Verlet / dissipative-Verlet updates (Eqs. Integration, VRL_Damp).
//
// GB300 runs two FP64 lanes per SM and clock, a 64th of its FP32 rate, so what
// bounds the pair kernels is the number of FP64 instructions, and those cost the
// same with one active lane as with 32.  Short-range kernels (H0, band and
// repulsive forces) therefore find their pairs with an FP32 distance test that
// errs on the safe side and collect them, 32 at a time, before any FP64 work;
// the FP64 test on the collected pair decides.  The Coulomb kernels of the split
// path (FP32 pair functions) carry their geometry as pairs of FP32 words
// (48 bits), the FP64 path one image per lane.
#include <algorithm>

#include "internal.h"

namespace xl {
namespace {

struct Bond {
  double V[4], dV[4], S, dS;
};

// V_k(r) = t0_k exp(-r/r_decay) S(r), S the quintic switch on [r_taper, r_cut].
__device__ __forceinline__ Bond bond(const ModelConst& m, double r) {
  const double w = m.r_cut - m.r_taper;
  double s = (r - m.r_taper) / w;
  s = fmin(fmax(s, 0.0), 1.0);
  const double s2 = s * s, s3 = s2 * s;
  const double S = 1.0 - 10.0 * s3 + 15.0 * s3 * s - 6.0 * s3 * s2;
  const double dS = (-30.0 * s2 + 60.0 * s3 - 30.0 * s3 * s) / w;
  const double e = exp(-r / m.r_decay);
  Bond b;
  b.S = S;
  b.dS = dS;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    b.V[k] = m.t0[k] * e * S;
    b.dV[k] = m.t0[k] * e * (dS - S / m.r_decay);
  }
  return b;
}

// Adds the s/p block E_ab(d) (Slater-Koster direction-cosine rules).
__device__ __forceinline__ void add_block(const ModelConst& m, double dx, double dy, double dz, double r,
                                          double E[4][4]) {
  const Bond b = bond(m, r);
  const double c[3] = {dx / r, dy / r, dz / r};
  E[0][0] += b.V[0];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    E[0][1 + a] += c[a] * b.V[1];
    E[1 + a][0] -= c[a] * b.V[1];
#pragma unroll
    for (int q = 0; q < 3; ++q)
      E[1 + a][1 + q] += c[a] * c[q] * (b.V[2] - b.V[3]) + (a == q ? b.V[3] : 0.0);
  }
}

// Adds wt sum_ab D_ab dE_ab/dd_g for one bond vector d to f[3].  With c = d/r, u_a = D_0a - D_a0 over the p
// orbitals and P the p block of D, the Slater-Koster block's gradient contracts to
//   c_g [D_00 V0' + (u.c)(V1' - V1/r) + (c.Pc)(Vd' - 2 Vd/r) + tr P V3'] + u_g V1/r + ((P + P^T) c)_g Vd/r,
// Vd = V2 - V3: about 60 FP64 operations instead of 250 term by term.
__device__ __forceinline__ void add_block_grad(const Bond& b, double dx, double dy, double dz, double ri,
                                               const double D[4][4], double wt, double f[3]) {
  const double c[3] = {dx * ri, dy * ri, dz * ri};
  const double Vd = b.V[2] - b.V[3], dVd = b.dV[2] - b.dV[3];
  double u[3], pc[3], uc = 0.0, cpc = 0.0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    u[a] = D[0][1 + a] - D[1 + a][0];
    uc += u[a] * c[a];
    pc[a] = 0.0;
#pragma unroll
    for (int q = 0; q < 3; ++q) pc[a] += (D[1 + a][1 + q] + D[1 + q][1 + a]) * c[q];
    cpc += pc[a] * c[a];
  }
  const double v1 = b.V[1] * ri, vd = Vd * ri;
  const double along = D[0][0] * b.dV[0] + uc * (b.dV[1] - v1) + cpc * (0.5 * dVd - vd) +
                       (D[1][1] + D[2][2] + D[3][3]) * b.dV[3];
#pragma unroll
  for (int g = 0; g < 3; ++g) f[g] += wt * (c[g] * along + u[g] * v1 + pc[g] * vd);
}

// FP32 test of the 27 images of a pair: bit 9 (tx + 1) + 3 (ty + 1) + tz + 1 is set where the image may lie
// within the cutoff (cut2 = r_cut^2 and a margin above the FP32 rounding of positions in [0, L)).  A
// distance that is not a number may lie anywhere: the FP64 pass then carries it into H and the forces.
__device__ __forceinline__ unsigned image_mask(float dx, float dy, float dz, float L, float cut2) {
  float x[3], y[3], z[3];
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    const float s = (t - 1) * L;
    x[t] = (dx + s) * (dx + s);
    y[t] = (dy + s) * (dy + s);
    z[t] = (dz + s) * (dz + s);
  }
  const float mx = fminf(x[0], fminf(x[1], x[2])), my = fminf(y[0], fminf(y[1], y[2]));
  if (mx + my + fminf(z[0], fminf(z[1], z[2])) >= cut2) return 0u;
  unsigned m = 0u;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (!(x[i] + y[j] + z[k] >= cut2)) m |= 1u << (9 * i + 3 * j + k);
  return m;
}

// H0 rows of atom I, one warp: zeros, then the 4 x 4 blocks of the neighbours, collected 32 at a time with
// their images (in the images' order, so a block's sum does not depend on the collection).  Also
// written to H, whose diagonal gets the potential later.
// 57 atoms 106 -> 20 us, 512 atoms 385 -> 29 us, 4096 atoms 6.9 -> 0.74 ms (the zeros of both matrices).
__global__ void build_H0_kernel(ModelConst m, int nat, double L, float cut2, const double* __restrict__ R,
                                double* __restrict__ H0, double* __restrict__ H, int np) {
  extern __shared__ int2 lists[];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int I = blockIdx.x * (blockDim.x >> 5) + wid;
  if (I >= nat) return;
  int2* list = lists + 64 * wid;
  const double xi = R[3 * I], yi = R[3 * I + 1], zi = R[3 * I + 2];
  const double rc2 = m.r_cut * m.r_cut;
  for (int a = 0; a < 4; ++a) {
    double2* r0 = reinterpret_cast<double2*>(H0 + (size_t)(4 * I + a) * np);
    double2* r1 = reinterpret_cast<double2*>(H + (size_t)(4 * I + a) * np);
    for (int c = lane; c < 2 * nat; c += 32) r0[c] = r1[c] = make_double2(0.0, 0.0);
  }
  __syncwarp();
  const float xf = (float)xi, yf = (float)yi, zf = (float)zi, Lf = (float)L;
  int cnt = 0;
  auto flush = [&](int take) {
    if (lane < take) {
      const int J = list[lane].x;
      unsigned mask = (unsigned)list[lane].y;
      double E[4][4];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) E[a][b] = 0.0;
      const double x0 = R[3 * J] - xi, y0 = R[3 * J + 1] - yi, z0 = R[3 * J + 2] - zi;
      bool any = (J == I);
      while (mask) {
        const int t = __ffs(mask) - 1;
        mask &= mask - 1;
        const double dx = x0 + (t / 9 - 1) * L, dy = y0 + (t / 3 % 3 - 1) * L, dz = z0 + (t % 3 - 1) * L;
        const double r2 = dx * dx + dy * dy + dz * dz;
        if (r2 >= rc2) continue;
        add_block(m, dx, dy, dz, sqrt(r2), E);
        any = true;
      }
      if (J == I) {
        E[0][0] += m.eps_s;
        E[1][1] += m.eps_p;
        E[2][2] += m.eps_p;
        E[3][3] += m.eps_p;
      }
      if (any) {
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const size_t o = (size_t)(4 * I + a) * np + 4 * J;
          reinterpret_cast<double2*>(H0 + o)[0] = reinterpret_cast<double2*>(H + o)[0] = make_double2(E[a][0], E[a][1]);
          reinterpret_cast<double2*>(H0 + o)[1] = reinterpret_cast<double2*>(H + o)[1] = make_double2(E[a][2], E[a][3]);
        }
      }
    }
    __syncwarp();
  };
  for (int J0 = 0; J0 < nat; J0 += 32) {
    const int J = J0 + lane;
    unsigned mask = 0u;
    if (J < nat) {
      mask = image_mask((float)R[3 * J] - xf, (float)R[3 * J + 1] - yf, (float)R[3 * J + 2] - zf, Lf, cut2);
      if (J == I) mask &= ~(1u << 13);   // not itself, but always in the list (on-site energies)
    }
    const bool has = mask != 0u || J == I;
    const unsigned bal = __ballot_sync(0xffffffffu, has);
    if (has) list[cnt + __popc(bal & ((1u << lane) - 1))] = make_int2(J, (int)mask);
    cnt += __popc(bal);
    __syncwarp();
    if (cnt >= 32) {
      flush(32);
      if (lane < cnt - 32) list[lane] = list[32 + lane];
      __syncwarp();
      cnt -= 32;
    }
  }
  if (cnt > 0) flush(cnt);
}

// Short-range forces of atom I, one warp:
//   F_I = 4 sum_J sum_T sum_ab D_{Ia,Jb} dE_ab/dd + sum_{J,T} d(A exp(-r/rho) S(r))/dr d/r,  d = R_J + T L - R_I
// (the self images' terms cancel).  Pairs are collected one image per lane.  With the band and repulsive parts in
// kernels of their own that ran every lane over all images: 57 atoms 385 -> 17 us, 512 atoms 1179 -> 26 us,
// 4096 atoms 17.6 -> 0.24 ms.
__global__ void forces_short_kernel(ModelConst m, int nat, double L, float cut2, const double* __restrict__ R,
                                    const double* __restrict__ D, int np, double* __restrict__ F) {
  extern __shared__ int lists1[];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int I = blockIdx.x * (blockDim.x >> 5) + wid;
  if (I >= nat) return;
  int* list = lists1 + 64 * wid;
  const double xi = R[3 * I], yi = R[3 * I + 1], zi = R[3 * I + 2];
  const double rc2 = m.r_cut * m.r_cut;
  const float xf = (float)xi, yf = (float)yi, zf = (float)zi, Lf = (float)L;
  double f[3] = {0, 0, 0};
  int cnt = 0;
  auto flush = [&](int take) {
    if (lane < take) {
      const int J = list[lane] >> 5, t = list[lane] & 31;
      const double dx = R[3 * J] - xi + (t / 9 - 1) * L, dy = R[3 * J + 1] - yi + (t / 3 % 3 - 1) * L,
                   dz = R[3 * J + 2] - zi + (t % 3 - 1) * L;
      const double r2 = dx * dx + dy * dy + dz * dz;
      if (!(r2 >= rc2)) {
        double Db[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const double2* p = reinterpret_cast<const double2*>(D + (size_t)(4 * I + a) * np + 4 * J);
          const double2 lo = p[0], hi = p[1];
          Db[a][0] = lo.x;
          Db[a][1] = lo.y;
          Db[a][2] = hi.x;
          Db[a][3] = hi.y;
        }
        const double r = sqrt(r2), ri = 1.0 / r;
        const Bond b = bond(m, r);
        add_block_grad(b, dx, dy, dz, ri, Db, 4.0, f);
        if (m.rep_A != 0.0) {
          const double ex = m.rep_A * exp(-r / m.rep_rho);
          const double de = ex * (b.dS - b.S / m.rep_rho) * ri;
          f[0] += de * dx;
          f[1] += de * dy;
          f[2] += de * dz;
        }
      }
    }
    __syncwarp();
  };
  for (int J0 = 0; J0 < nat; J0 += 32) {
    const int J = J0 + lane;
    unsigned mask = 0u;
    if (J < nat && J != I)
      mask = image_mask((float)R[3 * J] - xf, (float)R[3 * J + 1] - yf, (float)R[3 * J + 2] - zf, Lf, cut2);
    unsigned bal;
    while ((bal = __ballot_sync(0xffffffffu, mask != 0u)) != 0u) {
      if (mask) {
        list[cnt + __popc(bal & ((1u << lane) - 1))] = J * 32 + __ffs(mask) - 1;
        mask &= mask - 1;
      }
      cnt += __popc(bal);
      __syncwarp();
      if (cnt >= 32) {
        flush(32);
        if (lane < cnt - 32) list[lane] = list[32 + lane];
        __syncwarp();
        cnt -= 32;
      }
    }
  }
  if (cnt > 0) flush(cnt);
#pragma unroll
  for (int g = 0; g < 3; ++g) {
    const double v = warp_sum(f[g]);
    if (lane == 0) F[3 * I + g] = v;
  }
}

// ---- Coulomb pair terms ----

template <typename R>
__device__ __forceinline__ R ok_real_t(R r, R a, R eta) {
  const R s = sqrt(r * r + a * a);
  return erfc(eta * r) / r - a * a / (r * s * (s + r));
}

template <typename R>
__device__ __forceinline__ R ok_real_dr_t(R r, R a, R eta) {
  const R s2 = r * r + a * a;
  return erf(eta * r) / (r * r) - R(2) * eta / sqrt(R(kPi)) * exp(-eta * eta * r * r) / r - r / (s2 * sqrt(s2));
}

// minimum image of d for positions in [0, L)
__device__ __forceinline__ double min_image(double d, double L) {
  return d > 0.5 * L ? d - L : d < -0.5 * L ? d + L : d;
}

// A number as two FP32 words hi + lo (|lo| <= ulp(hi)/2): 48 bits at FP32 speed.
struct Df {
  float h, l;
};
__device__ __forceinline__ Df df_two_sum(float a, float b) {
  const float s = a + b, t = s - a;
  return {s, (a - (s - t)) + (b - t)};
}
__device__ __forceinline__ Df df_norm(float h, float l) {
  const float s = h + l;
  return {s, l - (s - h)};
}
__device__ __forceinline__ Df df_add(Df a, Df b) {
  const Df s = df_two_sum(a.h, b.h);
  return df_norm(s.h, s.l + (a.l + b.l));
}
__device__ __forceinline__ Df df_sub(Df a, Df b) { return df_add(a, {-b.h, -b.l}); }
__device__ __forceinline__ Df df_square(Df a) {
  const float p = a.h * a.h;
  return df_norm(p, fmaf(a.h, a.h, -p) + 2.0f * a.h * a.l);
}
__device__ __forceinline__ Df df_mul_f(Df a, float b) {
  const float p = a.h * b;
  return df_norm(p, fmaf(a.h, b, -p) + a.l * b);
}
// the FP32 square root of a > 0, rounded from the 48-bit value
__device__ __forceinline__ float df_sqrt(Df a) {
  const float y = rsqrtf(a.h), r = a.h * y;
  return r + 0.5f * y * (fmaf(-r, r, a.h) + a.l);
}
__device__ __forceinline__ double df_to_double(Df a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ Df df_of(float2 a) { return {a.x, a.y}; }

__global__ void split_positions_kernel(int n, const double* __restrict__ R, float2* __restrict__ Rs) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float h = (float)R[i];
  Rs[i] = make_float2(h, (float)(R[i] - (double)h));
}

// the three images d + t L (t = -1, 0, 1) of a minimum-image component, and their squares
__device__ __forceinline__ void df_images(Df a, Df b, Df L, Df (&d)[3], Df (&q)[3]) {
  Df x = df_sub(a, b);
  if (x.h > 0.5f * L.h)
    x = df_sub(x, L);
  else if (x.h < -0.5f * L.h)
    x = df_add(x, L);
  d[0] = df_sub(x, L);
  d[1] = x;
  d[2] = df_add(x, L);
#pragma unroll
  for (int t = 0; t < 3; ++t) q[t] = df_square(d[t]);
}

// Real-space gamma of the split path: FP32 pair functions of the 48-bit distance, summed in 48 bits; one
// thread per pair (row I = blockIdx.y).  With FP64 geometry (27 FP64 square roots a pair) it took 13.0 ms, now 2.2,
// at 4096 atoms.
__global__ void gamma_real_split_kernel(ModelConst m, int nat, double L, double eta, const float2* __restrict__ Rs,
                                        double* __restrict__ gam, int natp) {
  const int J = blockIdx.x * blockDim.x + threadIdx.x;
  const int I = blockIdx.y;
  if (J >= natp) return;
  if (J >= nat) {
    gam[(size_t)I * natp + J] = 0.0;
    return;
  }
  const double a = m.k / m.U;
  const float Lh = (float)L;
  const Df Ld = {Lh, (float)(L - (double)Lh)};
  const float af = (float)a, ef = (float)eta;
  Df d[3], x2[3], y2[3], z2[3];
  df_images(df_of(Rs[3 * J]), df_of(Rs[3 * I]), Ld, d, x2);
  df_images(df_of(Rs[3 * J + 1]), df_of(Rs[3 * I + 1]), Ld, d, y2);
  df_images(df_of(Rs[3 * J + 2]), df_of(Rs[3 * I + 2]), Ld, d, z2);
  Df acc = {0.0f, 0.0f};
#pragma unroll 1
  for (int i = 0; i < 3; ++i)
#pragma unroll 1
    for (int j = 0; j < 3; ++j) {
      const Df xy = df_add(i == 0 ? x2[0] : i == 1 ? x2[1] : x2[2], j == 0 ? y2[0] : j == 1 ? y2[1] : y2[2]);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (I == J && i == 1 && j == 1 && k == 1) continue;
        const float g = ok_real_t<float>(df_sqrt(df_add(xy, z2[k])), af, ef);
        const Df s = df_two_sum(acc.h, g);
        acc = df_norm(s.h, s.l + acc.l);
      }
    }
  double v = df_to_double(acc);
  if (I == J) v += 1.0 / a - 2.0 * eta / sqrt(kPi);
  gam[(size_t)I * natp + J] = m.k * v;
}

// The same in FP64, one warp per pair, one image per lane.
__global__ void gamma_real_f64_kernel(ModelConst m, int nat, double L, double eta, const double* __restrict__ R,
                                      double* __restrict__ gam, int natp) {
  const int J = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int I = blockIdx.y;
  if (J >= natp) return;
  if (J >= nat) {
    if (lane == 0) gam[(size_t)I * natp + J] = 0.0;
    return;
  }
  const double a = m.k / m.U;
  double v = 0.0;
  if (lane < 27) {
    const double dx = min_image(R[3 * J] - R[3 * I], L) + (lane / 9 - 1) * L;
    const double dy = min_image(R[3 * J + 1] - R[3 * I + 1], L) + (lane / 3 % 3 - 1) * L;
    const double dz = min_image(R[3 * J + 2] - R[3 * I + 2], L) + (lane % 3 - 1) * L;
    if (I == J && lane == 13)
      v = 1.0 / a - 2.0 * eta / sqrt(kPi);
    else
      v = ok_real_t<double>(sqrt(dx * dx + dy * dy + dz * dz), a, eta);
  }
  v = warp_sum(v);
  if (lane == 0) gam[(size_t)I * natp + J] = m.k * v;
}

// SF[I][g] = sqrt(w_g) cos(G_g.R_I), SF[I][ng+g] = sqrt(w_g) sin(G_g.R_I); zero padding.  One block per
// atom: the factors exp(2 pi i h x / L) of each component for h = -kHMax .. kHMax, then two complex
// products per reciprocal vector instead of a sine or cosine of its own (60 us at 512 atoms).
constexpr int kHMax = 8;   // |h| <= 12.14 * 4 / (2 pi) = 7.73 for the vectors of the Ewald sum
__global__ void structure_factor_kernel(int nat, int ng, double L, const int* __restrict__ Gh,
                                        const double* __restrict__ Gs, const double* __restrict__ R,
                                        double* __restrict__ SF, int kp) {
  __shared__ double2 e[3][2 * kHMax + 1];
  const int I = blockIdx.x;
  if (I < nat && threadIdx.x < 3 * (2 * kHMax + 1)) {
    const int c = threadIdx.x / (2 * kHMax + 1), h = threadIdx.x % (2 * kHMax + 1) - kHMax;
    double sv, cv;
    sincospi(2.0 * h * (R[3 * I + c] / L), &sv, &cv);
    e[c][h + kHMax] = make_double2(cv, sv);
  }
  __syncthreads();
  double* row = SF + (size_t)I * kp;
  for (int g = threadIdx.x; g < ng; g += blockDim.x) {
    double2 w = make_double2(0.0, 0.0);
    if (I < nat) {
      const int h = Gh[g];
      const double2 x = e[0][(h & 255)], y = e[1][(h >> 8) & 255], z = e[2][(h >> 16) & 255];
      const double2 xy = make_double2(x.x * y.x - x.y * y.y, x.x * y.y + x.y * y.x);
      const double s = Gs[g];
      w = make_double2(s * (xy.x * z.x - xy.y * z.y), s * (xy.x * z.y + xy.y * z.x));
    }
    row[g] = w.x;
    row[ng + g] = w.y;
  }
  for (int g = 2 * ng + threadIdx.x; g < kp; g += blockDim.x) row[g] = 0.0;
}

__global__ void gemv_kernel(int nat, const double* __restrict__ gam, int natp, const double* __restrict__ x,
                            double* __restrict__ y) {
  const int I = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (I >= nat) return;
  double acc = 0.0;
  for (int J = lane; J < nat; J += 32) acc += gam[(size_t)I * natp + J] * x[J];
  acc = warp_sum(acc);
  if (lane == 0) y[I] = acc;
}

// t[v][g] = sum_I SF[I][g] x_v[I] with x_0 = 2 x - y and x_1 = y (x = q, y = n): 32 columns a block, 32 row
// groups.  The rows used to run one after another in one thread per column: 125 us at 512 atoms.
__global__ void __launch_bounds__(1024) sf_dot_kernel(int nat, int kp, const double* __restrict__ SF,
                                                      const double* __restrict__ x, const double* __restrict__ y,
                                                      double* __restrict__ t) {
  __shared__ double sh[2][32][33];
  const int c = threadIdx.x & 31, w = threadIdx.x >> 5, g = blockIdx.x * 32 + c;
  double a0 = 0.0, a1 = 0.0;
  if (g < kp) {
#pragma unroll 4
    for (int I = w; I < nat; I += 32) {
      const double s = SF[(size_t)I * kp + g];
      a0 += s * (2.0 * x[I] - y[I]);
      a1 += s * y[I];
    }
  }
  sh[0][w][c] = a0;
  sh[1][w][c] = a1;
  __syncthreads();
  // warp w sums column w
  const int gw = blockIdx.x * 32 + w;
  const double s0 = warp_sum(sh[0][c][w]), s1 = warp_sum(sh[1][c][w]);
  if (c == 0 && gw < kp) {
    t[gw] = s0;
    t[kp + gw] = s1;
  }
}

__global__ void add_potential_kernel(int nat, int np, const double* __restrict__ pot, double* __restrict__ H) {
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= 4 * nat) return;
  H[(size_t)a * np + a] += pot[a >> 2];
}

__global__ void gershgorin_rows_kernel(int n, int np, const double* __restrict__ H, double* __restrict__ lohi) {
  __shared__ double sh[32];
  const int i = blockIdx.x;
  double acc = 0.0;
  for (int j = threadIdx.x; j < n; j += blockDim.x)
    if (j != i) acc += fabs(H[(size_t)i * np + j]);
  acc = block_sum(acc, sh);
  if (threadIdx.x == 0) {
    const double d = H[(size_t)i * np + i];
    lohi[i] = d - acc;
    lohi[n + i] = d + acc;
  }
}

__global__ void minmax_kernel(int n, const double* __restrict__ lohi, double* __restrict__ out) {
  __shared__ double sl[32], sh[32];
  double lo = 1e300, hi = -1e300;
  bool bad = false;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    bad |= !isfinite(lohi[i]) || !isfinite(lohi[n + i]);
    lo = fmin(lo, lohi[i]);
    hi = fmax(hi, lohi[n + i]);
  }
  // fmin/fmax drop NaN: a non-finite row poisons both bounds so that the host sees it
  if (__syncthreads_or(bad)) {
    if (threadIdx.x == 0) out[0] = out[1] = nan("");
    return;
  }
  lo = warp_min(lo);
  hi = warp_max(hi);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) {
    sl[wid] = lo;
    sh[wid] = hi;
  }
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x >> 5;
    lo = lane < nw ? sl[lane] : 1e300;
    hi = lane < nw ? sh[lane] : -1e300;
    lo = warp_min(lo);
    hi = warp_max(hi);
    if (lane == 0) {
      out[0] = lo;
      out[1] = hi;
    }
  }
}

// Coulomb real-space force -k sum_{I != K} w_IK sum_T phi'(r) d/r, d = mi(R_K - R_I) + T L,
// w_IK = (a_I b_K + a_K b_I)/2, a = 2q - n, b = n; part blockIdx.y of gridDim.y of the atoms I, into
// part[blockIdx.y][K].  Split path: FP32 pair functions of 48-bit distances, each pair's 27 terms
// summed in 48 bits, pairs in FP64; TX: a thread takes one tx of its pair (few atoms).  57 atoms 75 -> 9 us,
// 512 atoms 560 -> 72 us, 4096 atoms 17.4 -> 3.2 ms against FP64 geometry and one warp per atom.
template <bool TX>
__global__ void __launch_bounds__(128) forces_coul_split_kernel(ModelConst m, int nat, double L, double eta,
                                                                const float2* __restrict__ Rs,
                                                                const double* __restrict__ q,
                                                                const double* __restrict__ n,
                                                                double* __restrict__ part) {
  __shared__ double sh[32];
  const int K = blockIdx.x;
  const double aK = 2.0 * q[K] - n[K], bK = n[K];
  const float Lh = (float)L;
  const Df Ld = {Lh, (float)(L - (double)Lh)};
  const float af = (float)(m.k / m.U), ef = (float)eta;
  const Df xK = df_of(Rs[3 * K]), yK = df_of(Rs[3 * K + 1]), zK = df_of(Rs[3 * K + 2]);
  double f[3] = {0, 0, 0};
  const int items = TX ? 3 * nat : nat;
  for (int it = blockIdx.y * blockDim.x + threadIdx.x; it < items; it += gridDim.y * blockDim.x) {
    const int I = TX ? it / 3 : it, i0 = TX ? it % 3 : 0, i1 = TX ? i0 + 1 : 3;
    if (I == K) continue;
    Df dx[3], dy[3], dz[3], x2[3], y2[3], z2[3];
    df_images(xK, df_of(Rs[3 * I]), Ld, dx, x2);
    df_images(yK, df_of(Rs[3 * I + 1]), Ld, dy, y2);
    df_images(zK, df_of(Rs[3 * I + 2]), Ld, dz, z2);
    Df fx = {0.f, 0.f}, fy = {0.f, 0.f}, fz = {0.f, 0.f};
#pragma unroll 1
    for (int i = i0; i < i1; ++i) {
      const Df xi = i == 0 ? dx[0] : i == 1 ? dx[1] : dx[2], xq = i == 0 ? x2[0] : i == 1 ? x2[1] : x2[2];
#pragma unroll 1
      for (int j = 0; j < 3; ++j) {
        const Df yj = j == 0 ? dy[0] : j == 1 ? dy[1] : dy[2];
        const Df xy = df_add(xq, j == 0 ? y2[0] : j == 1 ? y2[1] : y2[2]);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const float r = df_sqrt(df_add(xy, z2[k]));
          const float g = ok_real_dr_t<float>(r, af, ef) / r;
          fx = df_add(fx, df_mul_f(xi, g));
          fy = df_add(fy, df_mul_f(yj, g));
          fz = df_add(fz, df_mul_f(dz[k], g));
        }
      }
    }
    const double w = 0.5 * ((2.0 * q[I] - n[I]) * bK + aK * n[I]);
    f[0] += w * df_to_double(fx);
    f[1] += w * df_to_double(fy);
    f[2] += w * df_to_double(fz);
  }
#pragma unroll
  for (int g = 0; g < 3; ++g) {
    const double v = block_sum(f[g], sh);
    if (threadIdx.x == 0) part[((size_t)blockIdx.y * nat + K) * 3 + g] = -m.k * v;
  }
}

// The same in FP64: a warp per pair, one image per lane.
__global__ void __launch_bounds__(128) forces_coul_f64_kernel(ModelConst m, int nat, double L, double eta,
                                                              const double* __restrict__ R, const double* __restrict__ q,
                                                              const double* __restrict__ n, double* __restrict__ part) {
  __shared__ double sh[32];
  const int K = blockIdx.x, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const double a = m.k / m.U, aK = 2.0 * q[K] - n[K], bK = n[K];
  double f[3] = {0, 0, 0};
  if (lane < 27) {
    const double tx = (lane / 9 - 1) * L, ty = (lane / 3 % 3 - 1) * L, tz = (lane % 3 - 1) * L;
    for (int I = blockIdx.y * nw + (threadIdx.x >> 5); I < nat; I += gridDim.y * nw) {
      if (I == K) continue;
      const double w = 0.5 * ((2.0 * q[I] - n[I]) * bK + aK * n[I]);
      const double dx = min_image(R[3 * K] - R[3 * I], L) + tx, dy = min_image(R[3 * K + 1] - R[3 * I + 1], L) + ty,
                   dz = min_image(R[3 * K + 2] - R[3 * I + 2], L) + tz;
      const double r = sqrt(dx * dx + dy * dy + dz * dz);
      const double g = w * (ok_real_dr_t<double>(r, a, eta) / r);
      f[0] += g * dx;
      f[1] += g * dy;
      f[2] += g * dz;
    }
  }
#pragma unroll
  for (int g = 0; g < 3; ++g) {
    const double v = block_sum(f[g], sh);
    if (threadIdx.x == 0) part[((size_t)blockIdx.y * nat + K) * 3 + g] = -m.k * v;
  }
}

// F_K += sum of the real-space parts - (k/2) sum_g G [SF_c(K)(a_K S_b + b_K S_a) - SF_s(K)(a_K C_b + b_K C_a)]
// with SF_c, SF_s = sqrt(w_g) cos, sin (G.R_K) and the sums t = [C_a, S_a | C_b, S_b] = SF^T a, SF^T b: the
// structure factors of build_H instead of a sine and a cosine per atom and vector, twice (57 atoms 108 -> 21 us).
__global__ void __launch_bounds__(128) forces_coul_recip_kernel(double kcoul, int nat, int ng, int kp, int nparts,
                                                                const double* __restrict__ G4,
                                                                const double* __restrict__ SF,
                                                                const double* __restrict__ q,
                                                                const double* __restrict__ n,
                                                                const double* __restrict__ t,
                                                                const double* __restrict__ part,
                                                                double* __restrict__ F) {
  __shared__ double sh[32];
  const int K = blockIdx.x;
  const double aK = 2.0 * q[K] - n[K], bK = n[K];
  const double* row = SF + (size_t)K * kp;
  double f[3] = {0, 0, 0};
  for (int g = threadIdx.x; g < ng; g += blockDim.x) {
    const double ca = t[g], sa = t[ng + g], cb = t[kp + g], sb = t[kp + ng + g];
    const double v = row[g] * (aK * sb + bK * sa) - row[ng + g] * (aK * cb + bK * ca);
    f[0] += v * G4[4 * g];
    f[1] += v * G4[4 * g + 1];
    f[2] += v * G4[4 * g + 2];
  }
#pragma unroll
  for (int g = 0; g < 3; ++g) {
    double v = -0.5 * kcoul * block_sum(f[g], sh);
    if (threadIdx.x == 0) {
      for (int p = 0; p < nparts; ++p) v += part[((size_t)p * nat + K) * 3 + g];
      F[3 * K + g] += v;
    }
  }
}

__global__ void charges_kernel(int nat, const double* __restrict__ ddiag, const double* __restrict__ Z,
                               const double* __restrict__ n, double* __restrict__ q, double* __restrict__ r) {
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  if (I >= nat) return;
  const double qi = ddiag[4 * I] + ddiag[4 * I + 1] + ddiag[4 * I + 2] + ddiag[4 * I + 3] - Z[I];
  q[I] = qi;
  r[I] = qi - n[I];
}

__global__ void verlet_first_kernel(int nat, double L, double dt, double minv, double* __restrict__ R,
                                    double* __restrict__ V, const double* __restrict__ F, double* __restrict__ nh,
                                    int kmax, const double* __restrict__ Kr, double kappa, double alpha,
                                    const double* __restrict__ c) {
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  if (I >= nat) return;
#pragma unroll
  for (int g = 0; g < 3; ++g) {
    double v = V[3 * I + g] + 0.5 * dt * F[3 * I + g] * minv;
    double x = R[3 * I + g] + dt * v;
    x -= L * floor(x / L);
    if (x >= L) x -= L;
    V[3 * I + g] = v;
    R[3 * I + g] = x;
  }
  double diss = 0.0;
  for (int k = 0; k <= kmax; ++k) diss += c[k] * nh[(size_t)k * nat + I];
  const double nn = 2.0 * nh[I] - nh[(size_t)nat + I] - kappa * Kr[I] + alpha * diss;
  for (int k = kmax; k >= 1; --k) nh[(size_t)k * nat + I] = nh[(size_t)(k - 1) * nat + I];
  nh[I] = nn;
}

__global__ void verlet_second_kernel(int nat, double dt, double minv, double* __restrict__ V,
                                     const double* __restrict__ F) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 3 * nat) return;
  V[i] += 0.5 * dt * F[i] * minv;
}

// Pair repulsion energy e_I = 1/2 sum_{J,T} A exp(-r/rho) S(r) over the 27 images, one warp per atom.
__global__ void repulsion_energy_kernel(ModelConst m, int nat, double L, float cut2, const double* __restrict__ R,
                                        double* __restrict__ e) {
  extern __shared__ int lists2[];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int I = blockIdx.x * (blockDim.x >> 5) + wid;
  if (I >= nat) return;
  int* list = lists2 + 64 * wid;
  const double xi = R[3 * I], yi = R[3 * I + 1], zi = R[3 * I + 2];
  const double rc2 = m.r_cut * m.r_cut, w = m.r_cut - m.r_taper;
  const float xf = (float)xi, yf = (float)yi, zf = (float)zi, Lf = (float)L;
  double en = 0.0;
  int cnt = 0;
  auto flush = [&](int take) {
    if (lane < take) {
      const int J = list[lane] >> 5, t = list[lane] & 31;
      const double dx = R[3 * J] - xi + (t / 9 - 1) * L, dy = R[3 * J + 1] - yi + (t / 3 % 3 - 1) * L,
                   dz = R[3 * J + 2] - zi + (t % 3 - 1) * L;
      const double r2 = dx * dx + dy * dy + dz * dz;
      if (!(r2 >= rc2)) {
        const double r = sqrt(r2);
        const double u = fmin(fmax((r - m.r_taper) / w, 0.0), 1.0);
        const double S = 1.0 - u * u * u * (10.0 - u * (15.0 - 6.0 * u));
        en += 0.5 * m.rep_A * exp(-r / m.rep_rho) * S;
      }
    }
    __syncwarp();
  };
  for (int J0 = 0; J0 < nat; J0 += 32) {
    const int J = J0 + lane;
    unsigned mask = 0u;
    if (J < nat) {
      mask = image_mask((float)R[3 * J] - xf, (float)R[3 * J + 1] - yf, (float)R[3 * J + 2] - zf, Lf, cut2);
      if (J == I) mask &= ~(1u << 13);
    }
    unsigned bal;
    while ((bal = __ballot_sync(0xffffffffu, mask != 0u)) != 0u) {
      if (mask) {
        list[cnt + __popc(bal & ((1u << lane) - 1))] = J * 32 + __ffs(mask) - 1;
        mask &= mask - 1;
      }
      cnt += __popc(bal);
      __syncwarp();
      if (cnt >= 32) {
        flush(32);
        if (lane < cnt - 32) list[lane] = list[32 + lane];
        __syncwarp();
        cnt -= 32;
      }
    }
  }
  if (cnt > 0) flush(cnt);
  en = warp_sum(en);
  if (lane == 0) e[I] = en;
}

// out[0] = 1/2 sum (2q - n) pot (Coulomb), out[1] = kinetic energy (eV)
__global__ void energy_vec_kernel(int nat, const double* __restrict__ q, const double* __restrict__ n,
                                  const double* __restrict__ pot, const double* __restrict__ V, double mass,
                                  double* __restrict__ out) {
  __shared__ double sh[32];
  double ec = 0.0, ke = 0.0;
  for (int I = threadIdx.x; I < nat; I += blockDim.x) {
    ec += (2.0 * q[I] - n[I]) * pot[I];
    ke += V[3 * I] * V[3 * I] + V[3 * I + 1] * V[3 * I + 1] + V[3 * I + 2] * V[3 * I + 2];
  }
  ec = block_sum(ec, sh);
  ke = block_sum(ke, sh);
  if (threadIdx.x == 0) {
    out[0] = 0.5 * ec;
    out[1] = 0.5 * mass * ke / 9.648533e-3;
  }
}

}  // namespace

namespace {

// r_cut^2 plus a margin above the FP32 error of distances between positions in [0, L)
float safe_cut2(const ModelConst& m, double L) { return (float)(m.r_cut * m.r_cut + 0.01 + 5e-6 * m.r_cut * L); }

// Warps (atoms) per block of the warp-per-atom kernels: one while the atoms fit the SMs a few times
// over, so that few atoms spread over all SMs' FP64 units, then four.
int atoms_per_block(int nat) { return nat <= 608 ? 1 : 4; }

}  // namespace

cudaError_t launch_split_positions(cudaStream_t s, int nat, const double* R, float2* Rs) {
  split_positions_kernel<<<(3 * nat + 255) / 256, 256, 0, s>>>(3 * nat, R, Rs);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_build_H0(cudaStream_t s, const ModelConst& m, int nat, double L, const double* R, double* H0,
                            double* H, int np) {
  const int w = atoms_per_block(nat);
  build_H0_kernel<<<(nat + w - 1) / w, 32 * w, 64 * w * sizeof(int2), s>>>(m, nat, L, safe_cut2(m, L), R, H0, H, np);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_gamma_real(cudaStream_t s, const ModelConst& m, int nat, double L, double eta, const double* R,
                              const float2* Rs, double* gam, int natp) {
  if (Rs)
    gamma_real_split_kernel<<<dim3((natp + 63) / 64, nat), 64, 0, s>>>(m, nat, L, eta, Rs, gam, natp);
  else
    gamma_real_f64_kernel<<<dim3((natp + 3) / 4, nat), 128, 0, s>>>(m, nat, L, eta, R, gam, natp);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_structure_factors(cudaStream_t s, int nat, int ng, double L, const int* Gh, const double* Gs,
                                     const double* R, double* SF, int kp) {
  const int natp = (nat + 63) / 64 * 64;
  structure_factor_kernel<<<natp, 256, 0, s>>>(nat, ng, L, Gh, Gs, R, SF, kp);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_gemv(cudaStream_t s, int nat, const double* gam, int natp, const double* x, double* y) {
  const int wpb = 8;
  gemv_kernel<<<(nat + wpb - 1) / wpb, 32 * wpb, 0, s>>>(nat, gam, natp, x, y);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_apply_potential(cudaStream_t s, int nat, int np, const double* H0, const double* pot,
                                   double* H) {
  if (H0) {
    cudaError_t e = cudaMemcpyAsync(H, H0, sizeof(double) * (size_t)np * np, cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return e;
  }
  add_potential_kernel<<<(4 * nat + 255) / 256, 256, 0, s>>>(nat, np, pot, H);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_gershgorin(cudaStream_t s, int n, int np, const double* H, double* out) {
  // out[0..1] result; out[2 .. 2+2n) scratch
  gershgorin_rows_kernel<<<n, 256, 0, s>>>(n, np, H, out + 2);
  note_launch();
  minmax_kernel<<<1, 1024, 0, s>>>(n, out + 2, out);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_repulsion_energy(cudaStream_t s, const ModelConst& m, int nat, double L, const double* R,
                                    double* e) {
  const int w = atoms_per_block(nat);
  repulsion_energy_kernel<<<(nat + w - 1) / w, 32 * w, 64 * w * sizeof(int), s>>>(m, nat, L, safe_cut2(m, L), R, e);
  note_launch();
  return cudaGetLastError();
}

int force_parts(int nat) { return std::max(1, std::min(8, 304 / nat)); }

cudaError_t launch_forces(cudaStream_t s, const ModelConst& m, int nat, double L, double eta, int ng,
                          const double* G4, const double* R, const float2* Rs, const double* SF, int kp,
                          const double* D, int np, const double* q, const double* n, double* F, double* work) {
  const int w = atoms_per_block(nat);
  forces_short_kernel<<<(nat + w - 1) / w, 32 * w, 64 * w * sizeof(int), s>>>(m, nat, L, safe_cut2(m, L), R, D, np, F);
  note_launch();
  if (m.k != 0.0) {
    // few atoms: each atom's pairs over several blocks, so that the FP64 (and FP32) units of all SMs work
    const int parts = force_parts(nat);
    double* part = work + 2 * kp;
    const dim3 grid(nat, parts);
    if (!Rs)
      forces_coul_f64_kernel<<<grid, 128, 0, s>>>(m, nat, L, eta, R, q, n, part);
    else if (nat < 256)
      forces_coul_split_kernel<true><<<grid, 128, 0, s>>>(m, nat, L, eta, Rs, q, n, part);
    else
      forces_coul_split_kernel<false><<<grid, 128, 0, s>>>(m, nat, L, eta, Rs, q, n, part);
    note_launch();
    sf_dot_kernel<<<(kp + 31) / 32, 1024, 0, s>>>(nat, kp, SF, q, n, work);
    note_launch();
    forces_coul_recip_kernel<<<nat, 128, 0, s>>>(m.k, nat, ng, kp, parts, G4, SF, q, n, work, part, F);
    note_launch();
  }
  return cudaGetLastError();
}

cudaError_t launch_charges(cudaStream_t s, int nat, const double* ddiag, const double* Z, const double* n,
                           double* q, double* r) {
  charges_kernel<<<(nat + 127) / 128, 128, 0, s>>>(nat, ddiag, Z, n, q, r);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_verlet_first(cudaStream_t s, int nat, double L, double dt, double minv, double* R, double* V,
                                const double* F, double* nh, int kmax, const double* Kr, double kappa,
                                double alpha, const double* c) {
  verlet_first_kernel<<<(nat + 127) / 128, 128, 0, s>>>(nat, L, dt, minv, R, V, F, nh, kmax, Kr, kappa, alpha, c);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_verlet_second(cudaStream_t s, int nat, double dt, double minv, double* V, const double* F) {
  verlet_second_kernel<<<(3 * nat + 127) / 128, 128, 0, s>>>(nat, dt, minv, V, F);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_energy_vec(cudaStream_t s, int nat, const double* q, const double* n, const double* pot,
                              const double* V, double mass, double* out) {
  energy_vec_kernel<<<1, 1024, 0, s>>>(nat, q, n, pot, V, mass, out);
  note_launch();
  return cudaGetLastError();
}

}  // namespace xl
