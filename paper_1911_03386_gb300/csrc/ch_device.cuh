// ch_device.cuh -- device helpers shared by the kernel translation units: block reductions,
// sample partials and finalisation, thread-block cluster access.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "ch_internal.h"

namespace chk {
namespace {

// Fixed-order block reduction of two FP64 sums (deterministic for a given block size).
__device__ __forceinline__ void block_sum2(double& a, double& b, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (lane == 0) {
    red[2 * warp] = a;
    red[2 * warp + 1] = b;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double sa = 0.0, sb = 0.0;
    for (int w = 0; w < nw; ++w) {
      sa += red[2 * w];
      sb += red[2 * w + 1];
    }
    a = sa;
    b = sb;
  }
}

// FP32 form: FP64 partial sums of the F and dF/dt densities over the band's nr rows (C
// tile rows 2..nr+1) with mu recomputed in FP64 from the stored field once per point.  A
// warp walks a strip of rows down a chunk of 31 columns, carrying three C rows and two mu
// rows in registers; lane 31 holds the column after the chunk, so east neighbours come
// from the next lane.  Fixed work split and order: deterministic.
template <typename T>
__device__ void band_partials_mu64(const DevView& v, const Tile& tl, int nx, int nr, const MemberParams& P,
                                   double2* slot, double* red) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const double a = P.a, bx = P.bx, by = P.by;
  // the stored field in FP64 (hi + lo for compensated members), read from global memory:
  // band row q of the tile is field row j0 - 2 + q (periodic)
  const T* Hg = static_cast<const T*>(v.C) + P.offset;
  const T* Lg = P.comp ? static_cast<const T*>(v.C) + P.lo_offset : nullptr;
  const int ny = P.ny;
  // field row of band row q (q from -1 to nr + 3, j0 - 3 .. j0 + nr + 1): one wrap at most
  auto at = [&](int q, int ii) {
    int j = tl.start - 2 + q;
    j = j < 0 ? j + ny : (j >= ny ? j - ny : j);
    const int64_t k = (int64_t)j * nx + ii;
    return Lg ? (double)Hg[k] + (double)Lg[k] : (double)Hg[k];
  };
  const int nchunk = (nx + 30) / 31;
  const int nstrip = max(1, nwarps / nchunk);
  const int hs = (nr + nstrip - 1) / nstrip;
  // unscaled sums: (C^2 - 1)^2, (D+x C)^2, (D+y C)^2, (D+x mu)^2, (D+y mu)^2 (the grid
  // spacings and prefactors are applied once per thread at the end)
  double sw = 0.0, sdx = 0.0, sdy = 0.0, smx = 0.0, smy = 0.0;
  for (int item = warp; item < nchunk * nstrip; item += nwarps) {
    const int k = item % nchunk, r0 = (item / nchunk) * hs, r1 = min(nr, r0 + hs);
    if (r0 >= r1) continue;
    const int i = (31 * k + lane) % nx;
    const bool own = lane < 31 && 31 * k + lane < nx;
    const int iw = i == 0 ? nx - 1 : i - 1, ie = i + 1 == nx ? 0 : i + 1;
    // C at tile row q in FP64, and its west / east neighbours (shuffles inside the chunk)
    auto cload = [&](int q) { return at(q, i); };
    auto mu_row = [&](int q, double cq, double cdn, double cup) {
      double w = __shfl_up_sync(full, cq, 1), e = __shfl_down_sync(full, cq, 1);
      if (lane == 0) w = at(q, iw);
      if (lane == 31) e = at(q, ie);
      return cq * (cq * cq - a) - bx * (e + w) - by * (cup + cdn);
    };
    const int q0 = r0 + 2;
    double cm = cload(q0 - 1), c0 = cload(q0), c1 = cload(q0 + 1), c2 = cload(q0 + 2);
    double mu0 = mu_row(q0, c0, cm, c1);
    double mu1 = mu_row(q0 + 1, c1, c0, c2);
    for (int r = r0; r < r1; ++r) {
      const double ce = __shfl_down_sync(full, c0, 1);
      const double mue = __shfl_down_sync(full, mu0, 1);
      if (own) {
        const double w = c0 * c0 - 1.0, gx = ce - c0, gy = c1 - c0, mx = mue - mu0, my = mu1 - mu0;
        sw += w * w;
        sdx += gx * gx;
        sdy += gy * gy;
        smx += mx * mx;
        smy += my * my;
      }
      if (r + 1 < r1) {  // advance: row q+3 enters, mu of row q+2
        const double c3 = cload(r + 5);
        const double mu2 = mu_row(r + 4, c2, c1, c3);
        c0 = c1;
        c1 = c2;
        c2 = c3;
        mu0 = mu1;
        mu1 = mu2;
      }
    }
  }
  const double hxi2 = 1.0 / (P.hx * P.hx), hyi2 = 1.0 / (P.hy * P.hy);
  double sF = 0.25 * sw + 0.5 * P.gamma * (hxi2 * sdx + hyi2 * sdy);
  double sD = hxi2 * smx + hyi2 * smy;
  block_sum2(sF, sD, red);
  if (threadIdx.x == 0) *slot = make_double2(sF, sD);
}

// Active flag and sample decision of a stencil-phase CTA.
__device__ __forceinline__ bool stencil_prologue(const Tile& tl, MemberState* st, const MemberParams& P, bool& sample) {
  const bool active = st->remaining > 0;
  if (tl.index == 0 && threadIdx.x == 0) st->active = active ? 1 : 0;
  sample = (st->step % P.every) == 0;
  return active;
}

__device__ __forceinline__ double* red_buffer(unsigned char* smem, size_t tile_bytes) {
  return reinterpret_cast<double*>(smem + ((tile_bytes + 15) & ~(size_t)15));
}

// The sample itself from the member's summed partials (sF, sD): F, dF/dt, beta, the series
// ring and the window average; then the step counter and horizon advance.
__device__ __forceinline__ void finalize_sums(const DevView& v, int member, MemberState* st, const MemberParams& P,
                                              double sF, double sD) {
  const int64_t n = st->step;
  if (n % P.every == 0) {
    const double hh = P.hx * P.hy;
    const double F = hh * sF;
    const double dFdt = -(hh * sD);
    const double t = (double)n * P.dt;
    const double beta = -(t / F) * dFdt;
    st->F = F;
    st->dFdt = dFdt;
    st->beta = beta;
    if (!isfinite(F) || !isfinite(dFdt)) st->nonfinite = 1;
    if (P.series_cap > 0) {
      double* s = v.series + ((size_t)member * P.series_cap + (size_t)(st->nsamples % P.series_cap)) * 4;
      s[0] = t;
      s[1] = F;
      s[2] = dFdt;
      s[3] = beta;
    }
    st->nsamples += 1;
    if (t >= P.t1) {
      st->beta_sum += beta;
      st->beta_count += 1;
    }
  }
  st->step = n + 1;
  if (st->remaining != kUnbounded) st->remaining -= 1;
}

// Sample finalisation of one member (called once per member and step by the column phase,
// after the stencil phase wrote the band partials): the partials summed in band order, then
// finalize_sums.
__device__ __forceinline__ void finalize_sample(const DevView& v, int member, MemberState* st, const MemberParams& P) {
  double sF = 0.0, sD = 0.0;
  if (st->step % P.every == 0) {
    for (int b = 0; b < P.nbands; ++b) {
      const double2 pr = v.partials[P.partial_base + b];
      sF += pr.x;
      sD += pr.y;
    }
  }
  finalize_sums(v, member, st, P, sF, sD);
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// Shared-memory address of p in CTA `rank` of the cluster.
__device__ __forceinline__ unsigned peer_addr(const void* p, unsigned rank) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}

__device__ __forceinline__ float ld_peer(unsigned addr, float) {
  float x;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x) : "r"(addr) : "memory");
  return x;
}
__device__ __forceinline__ double ld_peer(unsigned addr, double) {
  double x;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(x) : "r"(addr) : "memory");
  return x;
}

}  // namespace
}  // namespace chk
