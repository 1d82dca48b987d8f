// K1 with the slice profile: Gaussian RF pulses played as sub-steps against a balanced
// slice-select gradient, averaged over isochromats across the slice (Methods, "Pulse
// Sequence": Gaussian envelopes; "Reconstructions": the Bloch solver takes the slice
// profile into account).  The model (the paper gives no pulse parameters):
//   isochromat k of n_iso sits at u_k = extent ((k + 1/2)/n_iso - 1/2) slice thicknesses;
//   the pulse is n_sub hard sub-pulses with Gaussian weights w_s (sum 1), sub-step s
//   turns about the TR's RF axis by phi_n w_s (phi_n the signed flip, as in the
//   hard-pulse kernel) and then precesses about z by beta_k = 2 pi tbw u_k / n_sub;
//   a pre-winder and a rewinder of -n_sub/2 beta_k each balance the gradient;
//   the rest of the TR as in the hard-pulse recursion, per isochromat; the echo is the
//   mean of m_y over the isochromats (the x components cancel by the slice's mirror
//   symmetry, so the signal stays i * mean m_y).
//
// Mirror symmetry halves the isochromats: u_k = -u_{n_iso-1-k}, so the two see opposite
// precessions, and (m_x, m_y, m_z) -> (-m_x, m_y, m_z) maps one recursion to the other; the
// mean of m_y runs over k < n_iso / 2.  A lane carries two of them in packed float32 pairs
// (packed.cuh): 8 lanes per voxel for 32 isochromats, 4 voxels per warp, the 3-vector state
// and its ln T1 / ln T2 tangents in registers.  The relaxation over TE and over TR - TE act
// on the same state one after the other, so the state takes both as one step over TR; the
// echo, which only the first step reaches, is E2(TE) times the sum over the isochromats
// (plus its ln T2 source), applied once per voxel after the sum.  The pulse of a (TR,
// isochromat) pair does not depend on the voxel: mrstat_set_slice_profile composes each one
// once, in float64 on the host, into a 3 x 3 matrix (columns: the basis vectors pushed
// through pre-winder, sub-steps and rewinder); each block stages a chunk of TRs' matrices in
// shared memory and its lanes apply them.
//
// Bound by the FP32 pipe: per TR and isochromat pair 27 packed multiply-adds for the pulse
// on the state and both tangents and 13 for the relaxation.  At 224 x 224, 1120 TRs and 32
// isochromats: 1.63 ms with the tangents, 0.59 ms for m alone (5.86 and 5.61 ms with one
// lane per isochromat and the two decays).
#include <algorithm>
#include <cmath>

#include "internal.cuh"
#include "packed.cuh"

namespace mrstat {
namespace {

constexpr int kSliceThreads = 256;
constexpr int kSliceChunk = 16;  // TRs per staged chunk
constexpr int kSliceMaxSub = 64;
constexpr int kRotStride = 10;   // pairs per (TR, isochromat pair): 9 and padding to 16 bytes

// L lanes per voxel group (L = 1, 2, 4, 8 isochromat pairs), V voxels per lane sharing each
// loaded matrix; NCH 1: m only, 3: with both tangents.
template <int L, int NCH, int V>
__global__ void __launch_bounds__(kSliceThreads)
bloch_slice_kernel(const float* __restrict__ alpha, const uint8_t* __restrict__ mask,
                   const float2* __restrict__ rotg, int nv, int nq, float te, float tr, float m0z,
                   float4* __restrict__ D) {
  using pk::f2;
  constexpr int kVals = 4 * NCH;              // echo values of a TR quad
  constexpr int kHalves = L < 4 ? L : 4;      // lanes that share them after the exchanges
  constexpr int kKeep = kVals / kHalves;      // values a lane ends with: 4 / kHalves TRs
  __shared__ __align__(16) f2 rot[kSliceChunk * L * kRotStride];
  const int tid = threadIdx.x, lane = tid & 31;
  const int p = lane & (L - 1);  // this lane's isochromat pair
  const int j0 = ((blockIdx.x * kSliceThreads + tid) >> 5) * (V * 32 / L) + lane / L;
  const size_t cstride = (size_t)nq * nv;

  // over TR: m += (E - 1)(m - m_eq) with E - 1 from expm1f; d = dE/dln T.  Over TE the
  // transverse factor and its derivative, for the echo
  const f2 minus1 = pk::both(-1.f), zero = pk::both(0.f);
  f2 x1[V], x2[V], d1[V], d2[V], m[V][3], a[V][3], b[V][3];
  float x2e[V], d2e[V], norm[V];
  bool any = false;
#pragma unroll
  for (int w = 0; w < V; ++w) {
    const int j = j0 + w * (32 / L);
    const bool live = j < nv;
    const bool on = live && (mask == nullptr || mask[j] != 0);
    any |= on;
    float t1 = 1000.f, t2 = 100.f;
    if (live) {
      t1 = expf(alpha[j]);
      t2 = expf(alpha[nv + j]);
    }
    // a voxel outside the mask stands for zeros whatever its parameters are (NaN too)
    t1 = on ? t1 : 1000.f;
    t2 = on ? t2 : 100.f;
    const float x1s = expm1f(-tr / t1), x2s = expm1f(-tr / t2);
    x1[w] = pk::both(x1s);
    x2[w] = pk::both(x2s);
    d1[w] = pk::both(tr / t1 * (1.f + x1s));
    d2[w] = pk::both(tr / t2 * (1.f + x2s));
    x2e[w] = expm1f(-te / t2);
    d2e[w] = te / t2 * (1.f + x2e[w]);
    norm[w] = on ? 1.f / (float)(2 * L) : 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) m[w][i] = a[w][i] = b[w][i] = zero;
    m[w][2] = pk::both(m0z);
  }
  const bool work = __any_sync(0xffffffffu, any);  // a warp outside the mask only writes zeros

  const int ntr4 = 4 * nq;
  for (int n0 = 0; n0 < ntr4; n0 += kSliceChunk) {
    __syncthreads();  // the previous chunk's matrices are no longer read
    const int cnt = min(kSliceChunk, ntr4 - n0);
    {
      const float4* src = reinterpret_cast<const float4*>(rotg + (size_t)n0 * L * kRotStride);
      float4* dst = reinterpret_cast<float4*>(rot);
      for (int e = tid; e < cnt * L * kRotStride / 2; e += kSliceThreads) dst[e] = __ldg(src + e);
    }
    __syncthreads();
    for (int nq4 = 0; nq4 < cnt; nq4 += 4) {  // ntr4 and the quads are multiples of 4
      float v[V][kVals];
      if (work) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const ulonglong2* R2 = reinterpret_cast<const ulonglong2*>(rot + ((nq4 + u) * L + p) * kRotStride);
          f2 r[10];  // columns r[0..2], r[3..5], r[6..8]
#pragma unroll
          for (int e = 0; e < 5; ++e) {
            const ulonglong2 t = R2[e];
            r[2 * e] = t.x;
            r[2 * e + 1] = t.y;
          }
          auto turn = [&](f2 (&s)[3]) {
            f2 w[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) w[i] = pk::fma(r[i], s[0], pk::fma(r[3 + i], s[1], pk::mul(r[6 + i], s[2])));
            s[0] = w[0], s[1] = w[1], s[2] = w[2];
          };
#pragma unroll
          for (int w = 0; w < V; ++w) {
            turn(m[w]);
            const float2 my = pk::split(m[w][1]);
            v[w][NCH * u] = my.x + my.y;
            if (NCH > 1) {
              turn(a[w]);
              turn(b[w]);
              const float2 ay = pk::split(a[w][1]), by = pk::split(b[w][1]);
              v[w][NCH * u + 1] = ay.x + ay.y;
              v[w][NCH * u + 2] = by.x + by.y;
            }
            // decay over TR with the tangents' source terms (from the state before it)
            const f2 zm1 = pk::add(m[w][2], minus1);
            if (NCH > 1) {
              a[w][0] = pk::fma(x2[w], a[w][0], a[w][0]);
              a[w][1] = pk::fma(x2[w], a[w][1], a[w][1]);
              a[w][2] = pk::fma(x1[w], a[w][2], pk::fma(d1[w], zm1, a[w][2]));
              b[w][0] = pk::fma(x2[w], b[w][0], pk::fma(d2[w], m[w][0], b[w][0]));
              b[w][1] = pk::fma(x2[w], b[w][1], pk::fma(d2[w], m[w][1], b[w][1]));
              b[w][2] = pk::fma(x1[w], b[w][2], b[w][2]);
            }
            m[w][0] = pk::fma(x2[w], m[w][0], m[w][0]);
            m[w][1] = pk::fma(x2[w], m[w][1], m[w][1]);
            m[w][2] = pk::fma(x1[w], zm1, m[w][2]);
          }
        }
        // the quad's sums over the voxel's L lanes by halving: each exchange leaves a lane
        // with the half of the TRs its lane bit names; for L = 8 the lowest bit is added last
        if constexpr (L >= 2) {
#pragma unroll
          for (int w = 0; w < V; ++w) {
#pragma unroll
            for (int off = L / 2, n = kVals; n > kKeep; off >>= 1, n >>= 1) {
              const bool up = lane & off;
#pragma unroll
              for (int e = 0; e < n / 2; ++e) {
                const float send = up ? v[w][e] : v[w][n / 2 + e], keep = up ? v[w][n / 2 + e] : v[w][e];
                v[w][e] = keep + __shfl_xor_sync(0xffffffffu, send, off);
              }
            }
            if constexpr (L == 8) {
#pragma unroll
              for (int e = 0; e < kKeep; ++e) v[w][e] += __shfl_xor_sync(0xffffffffu, v[w][e], 1);
            }
          }
        }
      } else {
#pragma unroll
        for (int w = 0; w < V; ++w)
#pragma unroll
          for (int e = 0; e < kKeep; ++e) v[w][e] = 0.f;
      }
      if (L == 8 && (lane & 1)) continue;
      const int u0 = (L == 8 ? p >> 1 : p) * (4 / kHalves);  // this lane's first TR of the quad
#pragma unroll
      for (int w = 0; w < V; ++w) {
        const int j = j0 + w * (32 / L);
        if (j >= nv) continue;
        const size_t q = (size_t)((n0 + nq4) >> 2) * nv + j;
#pragma unroll
        for (int t = 0; t < 4 / kHalves; ++t) {
          const float sm = v[w][NCH * t] * norm[w];
          __stcs(reinterpret_cast<float*>(D + q) + u0 + t, fmaf(x2e[w], sm, sm));
          if (NCH > 1) {
            const float sa = v[w][NCH * t + 1] * norm[w], sb = v[w][NCH * t + 2] * norm[w];
            __stcs(reinterpret_cast<float*>(D + cstride + q) + u0 + t, fmaf(x2e[w], sa, sa));
            __stcs(reinterpret_cast<float*>(D + 2 * cstride + q) + u0 + t, fmaf(x2e[w], sb, fmaf(d2e[w], sm, sb)));
          }
        }
      }
    }
  }
}

// Isochromat pairs per voxel (lanes): the first half of the isochromats, two per lane; one
// or two isochromats fill one lane's pair with the same isochromat twice.
int slice_pairs(int n_iso) { return n_iso >= 4 ? n_iso / 4 : 1; }

template <int L, int NCH, int V>
cudaError_t launch_slice_t(const Plan& p, const float* alpha, const uint8_t* mask, float4* D, cudaStream_t st) {
  const int vpb = kSliceThreads / L * V;  // voxels per block
  bloch_slice_kernel<L, NCH, V><<<(p.nv + vpb - 1) / vpb, kSliceThreads, 0, st>>>(
      alpha, mask, reinterpret_cast<const float2*>(p.slice_rot), p.nv, p.nq, (float)p.te_ms, (float)p.tr_ms,
      p.inversion ? -1.f : 1.f, D);
  return cudaGetLastError();
}

// Without the tangents four voxels per lane share each loaded matrix (the shared-memory
// reads, five 16-byte loads per TR and lane, are then what one voxel per lane is bound by:
// 1.02 against 0.59 ms at 224 x 224, 1120 TRs, 32 isochromats), where that still leaves the
// SMs two warps per scheduler; with them the FP32 pipe is, and one voxel per lane keeps more
// warps in flight (1.63 against 1.75 ms with two).
template <int L>
cudaError_t launch_slice(const Plan& p, const float* alpha, const uint8_t* mask, float4* D, int nch, cudaStream_t st) {
  if (nch > 1) return launch_slice_t<L, 3, 1>(p, alpha, mask, D, st);
  const int64_t warps = ((int64_t)p.nv * L + 31) / 32;
  return warps >= 4 * 8 * (int64_t)p.sms ? launch_slice_t<L, 1, 4>(p, alpha, mask, D, st)
                              : launch_slice_t<L, 1, 1>(p, alpha, mask, D, st);
}

}  // namespace

cudaError_t launch_bloch_slice(const Plan& p, const float* alpha, const uint8_t* mask, float4* D, int nch,
                               cudaStream_t st) {
  if (p.nv == 0) return cudaSuccess;
  switch (slice_pairs(p.slice_iso)) {
    case 1: return launch_slice<1>(p, alpha, mask, D, nch, st);
    case 2: return launch_slice<2>(p, alpha, mask, D, nch, st);
    case 4: return launch_slice<4>(p, alpha, mask, D, nch, st);
    default: return launch_slice<8>(p, alpha, mask, D, nch, st);
  }
}

}  // namespace mrstat

using namespace mrstat;

extern "C" {

int mrstat_set_slice_profile(mrstat_plan* plan, const mrstat_slice_profile* prof) {
  MRSTAT_ABI_RANGE();
  Plan* p = reinterpret_cast<Plan*>(plan);
  if (p == nullptr) return fail(MRSTAT_ERR_INVALID_ARG, "NULL plan");
  DeviceGuard g(p->device);
  if (prof == nullptr) {
    p->slice_iso = 0;
    p->linearized = false;
    return MRSTAT_OK;
  }
  const int ni = prof->n_iso, ns = prof->n_sub;
  if (ni < 1 || ni > 32 || (ni & (ni - 1)) != 0 || ns < 1 || ns > kSliceMaxSub || !(prof->sigma > 0) ||
      !(prof->extent > 0) || !std::isfinite(prof->tbw))
    return fail(MRSTAT_ERR_INVALID_ARG, "slice profile: n_iso a power of two in 1..32, n_sub in 1..%d, "
                                        "sigma > 0, extent > 0", kSliceMaxSub);
  if (p->npar != 4) return fail(MRSTAT_ERR_UNSUPPORTED, "the slice-profile model has no B1 tangent");
  // Gaussian sub-pulse weights (sum 1), in float64
  std::vector<double> w(ns);
  double sum = 0.0;
  for (int s = 0; s < ns; ++s) {
    const double x = (s + 0.5) / ns - 0.5;
    w[s] = std::exp(-x * x / (2.0 * prof->sigma * prof->sigma));
    sum += w[s];
  }
  cudaError_t e = cudaSuccess;
  constexpr size_t kMaxPairs = 8;
  if (p->slice_rot == nullptr) e = dalloc(p, &p->slice_rot, (size_t)p->ntr_pad * kMaxPairs * kRotStride * 2);
  // the composed pulse of every (TR, isochromat): pre-winder, then per sub-step the RF
  // rotation by phi_n w_s about the TR's axis (the hard-pulse kernel's convention) and the
  // precession by beta_k, then the rewinder; in float64 from the plan's signed flips
  std::vector<float> phi(p->ntr_pad);
  if (e == cudaSuccess) e = cudaMemcpy(phi.data(), p->phi, phi.size() * sizeof(float), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "slice profile tables");
  // for the isochromats of the first half, laid out as pairs [TR][pair][9 + padding][2]
  const int pairs = slice_pairs(ni), half_iso = ni > 1 ? ni / 2 : 1;
  std::vector<float> rot((size_t)p->ntr_pad * pairs * kRotStride * 2, 0.f);
  for (int n = 0; n < p->ntr_pad; ++n)
    for (int kk = 0; kk < 2 * pairs; ++kk) {
      const int k = std::min(kk, half_iso - 1);
      const double u = prof->extent * ((k + 0.5) / ni - 0.5);
      const double beta = 2.0 * M_PI * prof->tbw * u / ns, half = -0.5 * ns * beta;
      const double cb = std::cos(beta), sb = std::sin(beta), ch = std::cos(half), sh = std::sin(half);
      for (int c = 0; c < 3; ++c) {
        double x = c == 0, y = c == 1, z = c == 2;
        double t = ch * x - sh * y;  // pre-winder
        y = sh * x + ch * y;
        x = t;
        for (int s = 0; s < ns; ++s) {
          const double ang = (double)phi[n] * (w[s] / sum), cn = std::cos(ang), sn = std::sin(ang);
          t = cn * y + sn * z;  // RF sub-pulse
          z = cn * z - sn * y;
          y = t;
          t = cb * x - sb * y;  // gradient precession
          y = sb * x + cb * y;
          x = t;
        }
        t = ch * x - sh * y;  // rewinder
        y = sh * x + ch * y;
        x = t;
        float* R = rot.data() + (((size_t)n * pairs + kk / 2) * kRotStride + 3 * c) * 2 + (kk & 1);
        R[0] = (float)x;
        R[2] = (float)y;
        R[4] = (float)z;
      }
    }
  e = cudaMemcpy(p->slice_rot, rot.data(), rot.size() * sizeof(float), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return cuda_fail(e, "slice profile tables");
  p->slice_iso = ni;
  p->slice_sub = ns;
  p->linearized = false;
  return MRSTAT_OK;
}

}  // extern "C"
