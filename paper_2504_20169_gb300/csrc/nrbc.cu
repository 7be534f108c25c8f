// Characteristic boundary targets (Sec. 4) and the final pass of the FP64 reductions.
#include <cfloat>

#include "lbm_internal.h"

namespace lbm {

// Rate dU/dt of one edge-band node (Sec. 4). U0: the node; U1, U2: the states one and two nodes
// inward along the normal (band layers or fluid moments); Va, Vb, Vc: three consecutive nodes of
// the same layer around it along the tangent with weights (ca, cb, cc) of the tangential
// derivative. PNR-LODI: Eq. (PNR) with Eq. (thermal_LODI_macro_evo); CBC relax: Eq. (CBC-Relax)
// with Eq. (thermal_CBC_macro_evo); viscous part zero. Differences in FP64, algebra in R.
//
// The launch is one short chain, and each FP64 instruction in it costs 64 cycles: so one division
// (1 / rho and 1 / (2 T) from 1 / (2 rho T)), factors that are powers of two applied to the sums in
// R, and 1 / (rho c) as c / (rho c^2). With P = rho T, c^2 = 2 T (gamma = 2): wave amplitudes
// w1,4 = T drho + rho dT -+ rho c du_n, w2 = T drho - rho dT, w3 = du_t, and back dP = (w1 + w4) / 2,
// du_n = (w4 - w1) / (2 rho c), drho = (dP + w2) / c^2, dT = (dP - T drho) / rho. With five
// divisions, FP64: 200 x 20 (D2Q17) 33.2 us a step, now 25.6; 300^2 51 -> 45 (FP32 within 2 %).
// The four stages stay one loop that reads the fluid's nodes again: unrolled, with those in
// registers (136 instead of 90), FP64 gains another 1 to 4 us, but the frame running beside it
// loses more (FP32: 512^2 41 -> 50 us, 2048^2 270 -> 287).
template <class R>
__device__ inline void char_rate(const BcParams& bc, int variant, double out, const Prim& U0d,
                                 const Prim& U1, const Prim& U2, const Prim& Va, const Prim& Vb,
                                 const Prim& Vc, double ca, double cb, double cc, bool xaxis,
                                 double kk[4]) {
  auto normal = [](double u0, double u1, double u2) { return R(fma(-4.0, u1, fma(3.0, u0, u2))); };
  const PrimT<R> U0 = to<R>(U0d);
  const R rho = U0.rho, un = U0.un, ut = U0.ut, T = U0.T;
  const R T2 = T + T, c = sqrt(T2), rc = rho * c;
  const R inv = R(1) / (rho * T2), irho = T2 * inv, iT2 = rho * inv;
  const R sgn = R(out);
  const bool in0 = (un - c) * sgn < R(0), in1 = un * sgn < R(0), in3 = (un + c) * sgn < R(0);
  R t0, t1, t2, t3;   // lambda_k w_k of the normal differences, in units of out / (2 r)
  {
    const R a = T * normal(U0d.rho, U1.rho, U2.rho), b = rho * normal(U0d.T, U1.T, U2.T);
    const R g = rc * normal(U0d.un, U1.un, U2.un);
    t0 = in0 ? R(0) : (un - c) * (a + b - g);
    t1 = in1 ? R(0) : un * (a - b);
    t2 = in1 ? R(0) : un * normal(U0d.ut, U1.ut, U2.ut);
    t3 = in3 ? R(0) : (un + c) * (a + b + g);
  }
  R scale = R(0.5 * out * bc.inv_r);
  if (variant != 0) {
    // B dU along the tangential axis (u_t advects; P_t = T rho_t + rho T_t; (2/D) T = T)
    auto along = [&](double va, double vb, double vc) { return R(ca * va + cb * vb + cc * vc); };
    const R dr = along(Va.rho, Vb.rho, Vc.rho), dn = along(Va.un, Vb.un, Vc.un);
    const R dt = along(Va.ut, Vb.ut, Vc.ut), dT = along(Va.T, Vb.T, Vc.T);
    const R br = ut * dr + rho * dt, bT = T * dt + ut * dT;
    const R a = T * br, b = rho * bT, g = rc * (ut * dn);
    const R w0 = a + b - g, w1 = a - b, w2 = T * irho * dr + ut * dt + dT, w3 = a + b + g;
    const R relax = R(1.0 + bc.relax_sign * (1.0 - bc.beta)), h = R(0.5 * out);
    t0 = in0 ? relax * w0 : h * t0 + w0;
    t1 = in1 ? relax * w1 : h * t1 + w1;
    t2 = in1 ? relax * w2 : h * t2 + w2;
    t3 = in3 ? relax * w3 : h * t3 + w3;
    scale = R(bc.inv_r);
  }
  const R dP = R(0.5) * (t0 + t3), drho = (dP + t1) * iT2;
  const R run = R(0.5) * (t3 - t0) * (c * inv), rT = (dP - T * drho) * irho;
  kk[0] = -double(scale * drho);
  kk[1] = -double(scale * (xaxis ? run : t2));
  kk[2] = -double(scale * (xaxis ? t2 : run));
  kk[3] = -double(scale * rT);
}

// All four stages of classical RK4 for the targets of one chunk of one edge band, in shared
// memory (fluid moments Ue frozen at time n), from the targets Vin of level n to V of level n + 1:
// two arrays, because blocks run in any order and a block's halo is another block's chunk.
// Block = one edge, tangential chunk [t0, t0 + T)
// plus a 4-node halo on each side where the chunk does not end the band; thread = (layer,
// position). Each stage shrinks the valid range by one node at a chunk cut, so the chunk's own
// nodes see exactly the values a full-band evaluation would. On a periodic y axis the W and E
// bands wrap around (central tangential differences everywhere, halo taken modulo Ly).
constexpr int kChunk = 32, kHalo = 4, kText = kChunk + 2 * kHalo;

// (nrbc_chunk is the per-block work; chunk = index over the four bands' chunks, sm = 16 M kText
// doubles of shared memory.)
template <class R>
__device__ __forceinline__ void nrbc_chunk(const Geom& g, const BcParams& bc,
                                           const double* __restrict__ Ue,
                                           const double* __restrict__ Se,
                                           const double* __restrict__ Vin,
                                           double* __restrict__ V, int chunk, double* sm) {
  const int M = g.M, Lx = g.Lx, Ly = g.Ly;
  const int cw = (Ly + kChunk - 1) / kChunk, cs = (Lx + kChunk - 1) / kChunk;
  int e, k = chunk;
  if (k < cw) e = 0;
  else if (k < 2 * cw) { e = 1; k -= cw; }
  else if (k < 2 * cw + cs) { e = 2; k -= 2 * cw; }
  else { e = 3; k -= 2 * cw + cs; }
  if (g.py && e >= 2) return;   // no S / N boundary on a periodic y axis
  const int len = e < 2 ? Ly : Lx;
  const int off = e == 0 ? 0 : e == 1 ? M * Ly : e == 2 ? 2 * M * Ly : 2 * M * Ly + M * Lx;
  const int ueoff = e == 0 ? 0 : e == 1 ? 2 * Ly : e == 2 ? 4 * Ly : 4 * Ly + 2 * Lx;
  const bool xaxis = e < 2;
  const double out = (e == 0 || e == 2) ? -1.0 : 1.0;
  const int t0 = k * kChunk;
  // along a periodic y axis the W / E bands are closed loops: the halo wraps around
  const bool wrap = g.py && e < 2;
  const int lo = wrap ? t0 - kHalo : max(0, t0 - kHalo);
  const int hi = wrap ? t0 + kChunk + kHalo : min(len, t0 + kChunk + kHalo);
  auto wr = [&](int tt) { return wrap ? ((tt % len) + len) % len : tt; };
  // shared state: [4 buffers][4 comps][M][kText] : V0, stage a, stage b, accumulator
  const int plane = M * kText;
  auto at = [&](int buf, int q, int j, int t) -> double& {
    return sm[(buf * 4 + q) * plane + (j - 1) * kText + (t - lo)];
  };
  const int tid = threadIdx.x;
  const int j = tid / kText + 1, t = lo + tid % kText;
  const bool live = j <= M && t < hi;
  if (live)
    for (int q = 0; q < 4; ++q) at(0, q, j, t) = Vin[q * g.nb + off + (j - 1) * len + wr(t)];
  __syncthreads();
  auto prim = [&](int buf, int jj, int tt) {
    Prim u;
    u.rho = at(buf, 0, jj, tt);
    const double ux = at(buf, 1, jj, tt), uy = at(buf, 2, jj, tt);
    u.un = xaxis ? ux : uy;
    u.ut = xaxis ? uy : ux;
    u.T = at(buf, 3, jj, tt);
    return u;
  };
  auto fluid = [&](int layer, int tt) {
    return load_prim(Ue, g.ne, ueoff + layer * len + wr(tt), xaxis);
  };
  const int variant = bc.edge[e];
  // Appendix PML source of this band position, mapped to (rho, u_x, u_y, T) rates at the
  // time-n state of the outermost fluid node: d rho = s_m, rho du = s_mom - u s_m,
  // (D/2) rho dT = s_E - u . s_mom + (u^2/2 - (D/2) T) s_m (D = 2); constant over the stages
  double src[4] = {0, 0, 0, 0};
  if ((bc.pml_source & 7) && live) {
    const int ns = 2 * (Lx + Ly);
    const int sb = (e == 0 ? 0 : e == 1 ? Ly : e == 2 ? 2 * Ly : 2 * Ly + Lx) + wr(t);
    const int ub = ueoff + wr(t);
    const double rho = Ue[ub], ux = Ue[g.ne + ub], uy = Ue[2 * g.ne + ub], T = Ue[3 * g.ne + ub];
    const double sm = Se[sb], sx = Se[ns + sb], sy = Se[2 * ns + sb], sE = Se[3 * ns + sb];
    src[0] = sm;
    src[1] = (sx - ux * sm) / rho;
    src[2] = (sy - uy * sm) / rho;
    src[3] = (sE - ux * sx - uy * sy + (0.5 * (ux * ux + uy * uy) - T) * sm) / rho;
    if (bc.pml_source & 8)   // the sign printed in Eq. (NSF-CHAR-PML)
      for (int q = 0; q < 4; ++q) src[q] = -src[q];
  }
  double kk[4] = {0, 0, 0, 0};
  for (int s = 1; s <= 4; ++s) {
    const int in_buf = s == 1 ? 0 : (s == 3 ? 2 : 1);  // V0, a, b, a
    const int slo = (!wrap && lo == 0) ? 0 : lo + s, shi = (!wrap && hi == len) ? len : hi - s;
    if (live && t >= slo && t < shi) {
      const Prim U0 = prim(in_buf, j, t);
      const Prim U1 = j >= 2 ? prim(in_buf, j - 1, t) : fluid(0, t);
      const Prim U2 = j >= 3 ? prim(in_buf, j - 2, t) : (j == 2 ? fluid(0, t) : fluid(1, t));
      int ta;
      double ca, cb, cc;
      if (!wrap && t == 0) { ta = 0; ca = -1.5; cb = 2.0; cc = -0.5; }
      else if (!wrap && t == len - 1) { ta = t - 2; ca = 0.5; cb = -2.0; cc = 1.5; }
      else { ta = t - 1; ca = -0.5; cb = 0.0; cc = 0.5; }
      Prim Va = U0, Vb = U0, Vc = U0;
      if (variant != 0) {
        Va = prim(in_buf, j, ta);
        Vb = prim(in_buf, j, ta + 1);
        Vc = prim(in_buf, j, ta + 2);
      }
      char_rate<R>(bc, variant, out, U0, U1, U2, Va, Vb, Vc, ca, cb, cc, xaxis, kk);
      for (int q = 0; q < 4; ++q) kk[q] += src[q];
    }
    __syncthreads();   // everyone has read the stage input before it is overwritten
    if (live && t >= slo && t < shi) {
      if (s < 4) {
        const int out_buf = s == 2 ? 2 : 1;            // a, b, a
        const double a = s == 3 ? 1.0 : 0.5, wgt = s == 1 ? 1.0 : 2.0;
        for (int q = 0; q < 4; ++q) {
          at(out_buf, q, j, t) = at(0, q, j, t) + a * kk[q];
          at(3, q, j, t) = (s == 1 ? 0.0 : at(3, q, j, t)) + wgt * kk[q];
        }
      } else if (t >= t0 && t < t0 + kChunk && t < len) {
        const double sixth = 1.0 / 6.0;
        for (int q = 0; q < 4; ++q)
          V[q * g.nb + off + (j - 1) * len + t] = at(0, q, j, t) + (at(3, q, j, t) + kk[q]) * sixth;
      }
    }
    __syncthreads();
  }
}

template <class R>
__global__ void kb_nrbc_rk4(const TgtDesc* __restrict__ d, const int* __restrict__ tab) {
  extern __shared__ double sm[];
  const int m = tab[2 * blockIdx.x], chunk = tab[2 * blockIdx.x + 1];
  const TgtDesc& t = d[m];
  nrbc_chunk<R>(t.g, t.bc, t.Ue, t.Se, t.Vin, t.V, chunk, sm);
}

void nrbc_shape(const Geom& g, int* chunks, int* threads, size_t* smem) {
  *chunks = 2 * ((g.Ly + kChunk - 1) / kChunk) + 2 * ((g.Lx + kChunk - 1) / kChunk);
  *threads = (g.M * kText + 31) / 32 * 32;
  *smem = sizeof(double) * 16 * g.M * kText;
}

cudaError_t launch_nrbc_batch(const TgtDesc* d, const int* tab, int n, bool fp32, int threads,
                              size_t smem, cudaStream_t s, cudaEvent_t begun) {
  if (n <= 0) return cudaSuccess;
  launch_begun(fp32 ? kb_nrbc_rk4<float> : kb_nrbc_rk4<double>, n, threads, smem, s, begun, d, tab);
  return cudaGetLastError();
}

// Final pass of the FP64 reductions: one block of 1024 threads; each thread folds whole
// 12-value records (contiguous, so a warp reads 32 consecutive records), then warp shuffles and
// one shared-memory round combine the 32 warps. Sums, except the slots flagged in min_mask
// (minimum).
__global__ void __launch_bounds__(1024) k_reduce_final(const double* __restrict__ partials, int n,
                                                      unsigned min_mask,
                                                      double* __restrict__ out) {
  __shared__ double sh[32][12];
  double a[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) a[k] = ((min_mask >> k) & 1u) ? DBL_MAX : 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double* r = partials + 12ll * i;
#pragma unroll
    for (int k = 0; k < 12; ++k) a[k] = ((min_mask >> k) & 1u) ? fmin(a[k], r[k]) : a[k] + r[k];
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
#pragma unroll
  for (int k = 0; k < 12; ++k)
    for (int o = 16; o > 0; o >>= 1) {
      const double t = __shfl_down_sync(0xffffffffu, a[k], o);
      a[k] = ((min_mask >> k) & 1u) ? fmin(a[k], t) : a[k] + t;
    }
  if (lane == 0)
    for (int k = 0; k < 12; ++k) sh[warp][k] = a[k];
  __syncthreads();
  if (warp == 0) {
    for (int k = 0; k < 12; ++k) {
      const bool mn = (min_mask >> k) & 1u;
      double b = lane < nwarps ? sh[lane][k] : (mn ? DBL_MAX : 0.0);
      for (int o = 16; o > 0; o >>= 1) {
        const double t = __shfl_down_sync(0xffffffffu, b, o);
        b = mn ? fmin(b, t) : b + t;
      }
      if (lane == 0) out[k] = b;
    }
  }
}

cudaError_t reduce_partials(const double* partials, int n, unsigned min_mask, double* out,
                            cudaStream_t st) {
  k_reduce_final<<<1, 1024, 0, st>>>(partials, n, min_mask, out);
  return cudaGetLastError();
}

}  // namespace lbm
