// The exact model's linearisation and products by re-running the Bloch recursion (hard
// pulses, no B1 map, ny <= 256): the default path of mrstat_linearize, mrstat_forward,
// mrstat_jvp, mrstat_jhw, mrstat_jhjv and of the checkpointed pair.  The paper evaluates the
// simulation inside every product (Algorithms 2 and 4); Supporting Information S2 gives the
// recursion.
//
// Why not stored time courses: at 224 x 224 and 1120 TRs they are 674 MB, 99 us of HBM per
// pass over them, and Re(J^H J) v passes twice (encode.cu: 111 + 126 us).  The recursion
// itself is cheap: per voxel and TR a rotation of m and both tangents (12 operations), one
// relaxation over TR (9; the relaxations over TE and TR - TE act on the same state one after
// the other) and no echo step at all, because the echo is E2(TE) times the rotated
// transverse component, a constant per voxel that the coefficients below absorb.  Two image
// rows per packed float32 pair (packed.cuh) halve the instructions, and everything a product
// needs beyond 19 floats per voxel and segment stays in registers.
//
// Linearisation: rx_states_kernel runs the recursion once per voxel, keeping the relaxation
// factors and the state before every seg-th TR.  The arrays are column-major ([ix][iy], the
// column stride nys even) so that a product's row pairs load as aligned float2.
//
// Products: block (column tile of 4, segment), 8 threads-rows per warp and column, each
// thread two row pairs; the phases come from a table per plan, copied asynchronously one chunk
// ahead into the warp's own ring.  With y, a, b the rotated m_y and tangents before the echo factor,
//     q = i (c m_e + rho (v0 a_e + v1 b_e)),  m_e = E y, a_e = E a, b_e = E b + D y,
//       = Q0 y + Q1 a + Q2 b                       (E = E2(TE), D = dE/dln T2; complex Q)
//     A[n][ix] = sum_iy Ey[n][iy] q_n(iy),          Ey[n][iy] = roots[(ky iy) mod ny]
//     Z_c = sum_n y_c[n] conj(Ey[n]) W[n][ix],      W = nx A (J^H J v) or the given rows
// and the gradient follows from E Z0, E Z1, E Z2 + D Z0.  TRs go in chunks (2 for J^H J v,
// whose echoes stay in registers until the block's sums stand, 8 for the sums alone, 4 for the
// adjoint, which needs no barrier): one barrier per chunk, the sums over the warps formed by every warp for itself.  The segments of a tile are
// the blocks of a cluster and add their gradients through distributed shared memory.
//
// Work: 41 packed multiply-adds per row pair and TR for Re(J^H J) v (68 us of the FP32 pipe at
// 224 x 224, 1120 TRs), 31 for the half products.  No single limit binds: counters show the
// pipe busy on 52 % (Re(J^H J) v) to 59 % (J.v) of the cycles (a packed instruction holds it for
// two) with 11-12 warps per SM, and the warps' stalls spread over the pipe (1.1-1.6 per
// instruction issued), fixed latencies (1.3-1.4), the chunks' barriers (0.8-1.0) and shared
// memory (0.3-0.9).  128 registers a thread (the state, factors, coefficients and sums of four
// rows) allow two blocks per SM.  Measured at that size, against the stored time courses:
// linearisation 50 us (120-180), J.v 92 (111 + 3), Re(J^H w) 92 (126), Re(J^H J) v 143 (241 in
// three launches), signal 29 + 49 (73 + 3 + 68).  Tried: two columns per block (129 / 131 / 177 us: the phases serve
// fewer threads), phases computed in the kernel instead of copied (106 / 103 / 158).
#include <algorithm>

#include <cooperative_groups.h>

#include "internal.cuh"
#include "packed.cuh"
#include "reduce.cuh"

namespace mrstat {
namespace {

using pk::f2;

enum { RX_JV = 0, RX_JHW = 1, RX_JHJV = 2 };

constexpr int kTX = 4;            // columns per block
constexpr int kLR = 32 / kTX;     // row-pair lanes per warp
constexpr int kRP = 2;            // row pairs per thread
constexpr int kMaxNy = 256;
constexpr int kMaxThreads = kMaxNy / (2 * kRP) * kTX;
constexpr int kMaxWarps = kMaxThreads / 32;
constexpr int kMaxSegments = 8;
constexpr int kWP = kLR * kRP;    // row pairs of a warp
__host__ __device__ constexpr int chunk_of(int mode) { return mode == RX_JHJV ? 2 : (mode == RX_JV ? 8 : 4); }
constexpr int kFac = 6;           // x1, x2, d1, d2 over TR; E, D over TE
constexpr int kStage = 512;       // TRs of the pulse table staged by the states kernel
constexpr int kTabs = 128;        // TRs of the tables staged by the product kernels (a multiple of 8)

int block_warps(int ny) { return (ny + 2 * kLR * kRP - 1) / (2 * kLR * kRP); }

// ---------------------------------------------------------------------------
// linearisation: factors and segment states, rho and the mask
// ---------------------------------------------------------------------------
// NCH 1: m only (2 floats per state), 3: with both tangents (6).  One voxel per thread,
// consecutive threads down a column.  The TRs' (cos, sin) come through shared memory, a
// kStage of TRs at a time: read from global memory as the recursion goes, every fourth TR
// waits for an L2 access (157 clocks per TR for a chain of about 20: 118 us with the tangents
// and 86 for m alone at 224 x 224, 1120 TRs; 50 and 29 from shared memory).
template <int NCH>
__global__ void __launch_bounds__(128)
rx_states_kernel(const float* __restrict__ alpha, const uint8_t* __restrict__ mask, const float2* __restrict__ cs,
                 int nx, int ny, int nys, int nv, int ntr, int seg, int nseg, float te, float tr, float m0z,
                 float* __restrict__ fac, float* __restrict__ st, float2* __restrict__ rho, float* __restrict__ maskf) {
  __shared__ __align__(16) float2 scs[kStage];
  const size_t nvp = (size_t)nx * nys;
  // threads past the last column repeat the last voxel's work (they meet the barriers) and
  // store nothing
  const int e0 = blockIdx.x * blockDim.x + threadIdx.x;
  const bool own = e0 < (int)nvp;
  const int e = own ? e0 : (int)nvp - 1;
  const int ix = e / nys, iy = e - ix * nys;
  const bool in = own && iy < ny;  // the padding row of an odd ny is no voxel
  const int j = (iy < ny ? iy : 0) * nx + ix;
  // a voxel outside the mask stands for zeros whatever its parameters are (NaN too)
  const bool count = in && (mask == nullptr || mask[j]);
  const float t1 = count ? expf(alpha[j]) : 1000.f, t2 = count ? expf(alpha[nv + j]) : 100.f;
  // E - 1 by expm1f: float32 keeps the small per-TR change of long T1/T2
  const float x1 = expm1f(-tr / t1), x2 = expm1f(-tr / t2), x2e = expm1f(-te / t2);
  const float d1 = tr / t1 * (1.f + x1), d2 = tr / t2 * (1.f + x2);
  const float fv[kFac] = {x1, x2, d1, d2, 1.f + x2e, te / t2 * (1.f + x2e)};
#pragma unroll
  for (int k = 0; k < kFac; ++k)
    if (own) fac[k * nvp + e] = fv[k];
  if (in) {
    rho[j] = count ? make_float2(alpha[2 * (size_t)nv + j], alpha[3 * (size_t)nv + j]) : make_float2(0.f, 0.f);
    if (maskf != nullptr) maskf[j] = count ? 1.f : 0.f;
  }
  constexpr int NS = NCH > 1 ? 6 : 2;
  float my = 0.f, mz = m0z, ay = 0.f, az = 0.f, by = 0.f, bz = 0.f;
  float* out = st + e;
  auto keep = [&]() {
    if (!own) return;
    out[0] = my;
    out[nvp] = mz;
    if (NCH > 1) {
      out[2 * nvp] = ay;
      out[3 * nvp] = az;
      out[4 * nvp] = by;
      out[5 * nvp] = bz;
    }
    out += NS * nvp;
  };
  keep();
  // whole segments before the last one; a voxel outside the mask keeps its first state
  const int nend = (nseg - 1) * seg;
  int next = seg;  // the TR before which the next state is kept
  for (int na = 0; na < nend; na += kStage) {
    __syncthreads();
    for (int i = threadIdx.x; i < min(kStage, nend - na) / 2; i += blockDim.x)  // seg is a multiple of 4
      reinterpret_cast<float4*>(scs)[i] = __ldg(reinterpret_cast<const float4*>(cs + na) + i);
    __syncthreads();
    const int ne = min(kStage, nend - na);
    for (int n0 = 0; n0 < ne; n0 += 4) {
      if (count) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float c = scs[n0 + k].x, s = scs[n0 + k].y;
          float t = c * my + s * mz;
          mz = c * mz - s * my;
          my = t;
          if (NCH > 1) {
            t = c * ay + s * az;
            az = c * az - s * ay;
            ay = t;
            t = c * by + s * bz;
            bz = c * bz - s * by;
            by = t;
          }
          const float zm1 = mz - 1.f;
          if (NCH > 1) {
            ay = fmaf(x2, ay, ay);
            az = fmaf(x1, az, fmaf(d1, zm1, az));
            by = fmaf(x2, by, fmaf(d2, my, by));
            bz = fmaf(x1, bz, bz);
          }
          my = fmaf(x2, my, my);
          mz = fmaf(x1, zm1, mz);
        }
      }
      if (na + n0 + 4 == next) {
        keep();
        next += seg;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// products
// ---------------------------------------------------------------------------
struct RxArgs {
  const float* fac;       // [6][nvp]
  const float* st;        // [nseg][ns][nvp], ns 6 or (m alone) 2
  int ns;
  const float* v;         // J.v, J^H J v: [4][nv]; NULL: the signal (c = rho)
  const float2* rho;      // rho * mask, [nv]
  const float* maskf;     // [nv] (unused by the signal)
  const float4* csp;      // [ntr_pad][2]
  const int* kyi;
  const float4* etab;     // [ny][16 warps]: (Re, Re, Im, Im) of Ey for ky and a pair of rows
  const float2* wt;       // J^H w: [ntr_pad][nx]
  int nx, ny, nys, nv, ntr, ntr_pad, seg, nseg, tiles;
  float scale;
  float2* A;              // J.v: [ntr][nx]
  float* g;               // [4][nv]
  unsigned* ticket;       // zero between launches
  double* red;            // [2 blocks] per-block inner products
  double *vdot, *vv;      // <v, g>, <v, v> or NULL
  const int* gate;
};

__device__ __forceinline__ void copy16(void* dst, const void* src, bool on) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(on ? 16 : 0)
               : "memory");
}

__device__ __forceinline__ f2 load2(const float* p, bool on) {
  if (!on) return 0ull;
  const float2 t = *reinterpret_cast<const float2*>(p);
  return pk::make(t.x, t.y);
}

template <int NCH, int MODE>
__global__ void __launch_bounds__(kMaxThreads, 2)
rx_product_kernel(const __grid_constant__ RxArgs P) {
  if (P.gate != nullptr && *P.gate == 0) return;
  constexpr int CT = chunk_of(MODE);  // TRs per chunk
  extern __shared__ float4 smem4[];
  const int nthr = blockDim.x, W = nthr >> 5;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, lx = lane % kTX, lr = lane / kTX;
  // the warp's own phases, two chunks: [2][CT][kWP]
  float4* ering = smem4 + warp * (2 * CT * kWP);
  const int nx = P.nx, ny = P.ny, nys = P.nys, nv = P.nv;
  const size_t nvp = (size_t)nx * nys;
  const int tile = blockIdx.x / P.nseg, sg = blockIdx.x - tile * P.nseg;  // a cluster: a tile's segments
  const int na = sg * P.seg, ne = min(P.ntr, na + P.seg);
  const int ix = tile * kTX + lx;
  // the tables of kTabs TRs: (c, c, s, s), (-s, -s) of the pulse, ky and (J^H w) W's rows
  float2* wtab = reinterpret_cast<float2*>(smem4 + W * (2 * CT * kWP));                 // [kTabs][kTX]
  float4* ctab = reinterpret_cast<float4*>(wtab + (MODE == RX_JHW ? kTabs * kTX : 0));  // [kTabs]
  float2* ntab = reinterpret_cast<float2*>(ctab + kTabs);                               // [kTabs]
  int* ktab = reinterpret_cast<int*>(ntab + kTabs);              // [kTabs]
  constexpr int NV = 2 * CT * kTX;                               // sums of a chunk: (TR, Re / Im, column)
  float* part = reinterpret_cast<float*>(ktab + kTabs);          // [2][NV][kMaxWarps], zero past W
  // J^H J v: the thread's coefficients, three (Re, Im) pairs of each row pair (registers hold
  // the state, the echoes of a chunk and the sums)
  ulonglong2* qtab = reinterpret_cast<ulonglong2*>(part + 2 * NV * kMaxWarps) + tid;  // [3 kRP][kMaxThreads]
  // the segment's gradient, read by the cluster: [4][rows][kTX]
  const int rows = W * kWP * 2;
  float* gbuf = part + (MODE == RX_JHW ? 0 : 2 * NV * kMaxWarps) +
                (MODE == RX_JHJV ? 3 * kRP * kMaxThreads * (int)(sizeof(ulonglong2) / sizeof(float)) : 0);
  if (MODE != RX_JHW)
    for (int i = tid; i < 2 * NV * kMaxWarps; i += nthr) part[i] = 0.f;

  int r0[kRP], ci[kRP];
  bool on[kRP];  // the pair's first row exists; its second may be the padding row
  f2 x1[kRP], x2[kRP], my[kRP], mz[kRP];
  f2 d1[kRP], d2[kRP], ay[kRP], az[kRP], by[kRP], bz[kRP];
  f2 qr0[kRP], qi0[kRP], qr1[kRP], qi1[kRP], qr2[kRP], qi2[kRP];
  bool live = false;  // some voxel of the thread counts
#pragma unroll
  for (int k = 0; k < kRP; ++k) {
    const int pr = (warp * kRP + k) * kLR + lr;
    r0[k] = 2 * pr;
    on[k] = r0[k] < ny && ix < nx;
    ci[k] = ix * nys + r0[k];
    const float* f = P.fac + ci[k];
    const float* s = P.st + (size_t)sg * P.ns * nvp + ci[k];
    x1[k] = load2(f, on[k]);
    x2[k] = load2(f + nvp, on[k]);
    my[k] = load2(s, on[k]);
    mz[k] = load2(s + nvp, on[k]);
    if (NCH > 1) {
      d1[k] = load2(f + 2 * nvp, on[k]);
      d2[k] = load2(f + 3 * nvp, on[k]);
      ay[k] = load2(s + 2 * nvp, on[k]);
      az[k] = load2(s + 3 * nvp, on[k]);
      by[k] = load2(s + 4 * nvp, on[k]);
      bz[k] = load2(s + 5 * nvp, on[k]);
    }
    float c[2][6];  // the rows' coefficients: (qr, qi) of y, a, b
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const bool o = on[k] && r0[k] + h < ny;
      // a row past the image reads row 0 of its own column: a NaN in v stays in its column
      const int j = o ? (r0[k] + h) * nx + ix : min(ix, nx - 1);
      float2 rh = make_float2(0.f, 0.f);
      if (MODE != RX_JHW) rh = o ? P.rho[j] : rh;
      const float e = o ? P.fac[4 * nvp + ci[k] + h] : 0.f;
      if (MODE == RX_JHW) {
        live |= o && P.maskf[j] != 0.f;
      } else if (NCH == 1) {
        live |= rh.x != 0.f || rh.y != 0.f;
        c[h][0] = -rh.y * e;
        c[h][1] = rh.x * e;
      } else {
        const float m = o ? P.maskf[j] : 0.f;
        live |= m != 0.f;
        const float d = o ? P.fac[5 * nvp + ci[k] + h] : 0.f;
        const float v0 = P.v[j], v1 = P.v[(size_t)nv + j];
        const float v2 = P.v[2 * (size_t)nv + j] * m, v3 = P.v[3 * (size_t)nv + j] * m;
        c[h][0] = -(v3 * e + rh.y * v1 * d);
        c[h][1] = v2 * e + rh.x * v1 * d;
        c[h][2] = -rh.y * e * v0;
        c[h][3] = rh.x * e * v0;
        c[h][4] = -rh.y * e * v1;
        c[h][5] = rh.x * e * v1;
      }
    }
    if (MODE == RX_JHJV) {
#pragma unroll
      for (int i = 0; i < 3; ++i)
        qtab[(3 * k + i) * kMaxThreads] = make_ulonglong2(pk::make(c[0][2 * i], c[1][2 * i]),
                                                   pk::make(c[0][2 * i + 1], c[1][2 * i + 1]));
    } else if (MODE == RX_JV) {
      qr0[k] = pk::make(c[0][0], c[1][0]);
      qi0[k] = pk::make(c[0][1], c[1][1]);
      if (NCH > 1) {
        qr1[k] = pk::make(c[0][2], c[1][2]);
        qi1[k] = pk::make(c[0][3], c[1][3]);
        qr2[k] = pk::make(c[0][4], c[1][4]);
        qi2[k] = pk::make(c[0][5], c[1][5]);
      }
    }
  }
  live = __any_sync(0xffffffffu, live);  // a warp outside the mask only keeps the barriers
  __syncthreads();

  // tables of the TRs [n0, n0 + kTabs): ky -1 past the segment, whose phases are zero
  auto tables = [&](int n0) {
    const int cnt = min(kTabs, ne - n0);
    for (int i = tid; i < kTabs; i += nthr) {
      ktab[i] = i < cnt ? __ldg(P.kyi + n0 + i) : -1;
      const bool in = n0 + i < P.ntr_pad;  // no rotation past the train
      ctab[i] = in ? __ldg(P.csp + 2 * (n0 + i)) : make_float4(1.f, 1.f, 0.f, 0.f);
      ntab[i] = in ? __ldg(reinterpret_cast<const float2*>(P.csp + 2 * (n0 + i) + 1)) : make_float2(0.f, 0.f);
    }
    if (MODE == RX_JHW)
      for (int i = tid; i < kTabs * kTX; i += nthr) {  // zero past the segment
        const int n = n0 + i / kTX, col = tile * kTX + i % kTX;
        wtab[i] = i < cnt * kTX && col < nx ? __ldg(P.wt + (size_t)n * nx + col) : make_float2(0.f, 0.f);
      }
  };
  // phases of the chunk at table position i0 (half a warp per TR), copied asynchronously
  auto phases = [&](int buf, int i0) {
    const int e = lane % kWP, half = lane / kWP;
#pragma unroll
    for (int i = 0; i < CT; i += 32 / kWP) {
      const int ky = ktab[i0 + i + half];
      copy16(ering + (buf * CT + i + half) * kWP + e, P.etab + (size_t)max(ky, 0) * (W * kWP) + warp * kWP + e, ky >= 0);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  f2 z[3][2][kRP];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int k = 0; k < kRP; ++k) z[c][0][k] = z[c][1][k] = 0ull;
  const f2 minus1 = pk::both(-1.f);
  auto turn = [](f2& y, f2& zc, f2 c, f2 s, f2 ms) {
    const f2 t = pk::fma(c, y, pk::mul(s, zc));
    zc = pk::fma(c, zc, pk::mul(ms, y));
    y = t;
  };
  auto rotate = [&](int k, f2 c, f2 s, f2 ms) {
    turn(my[k], mz[k], c, s, ms);
    if (NCH > 1) {
      turn(ay[k], az[k], c, s, ms);
      turn(by[k], bz[k], c, s, ms);
    }
  };
  auto decay = [&](int k) {
    const f2 zm1 = pk::add(mz[k], minus1);
    if (NCH > 1) {
      ay[k] = pk::fma(x2[k], ay[k], ay[k]);
      az[k] = pk::fma(x1[k], az[k], pk::fma(d1[k], zm1, az[k]));
      by[k] = pk::fma(x2[k], by[k], pk::fma(d2[k], my[k], by[k]));
      bz[k] = pk::fma(x1[k], bz[k], bz[k]);
    }
    my[k] = pk::fma(x2[k], my[k], my[k]);
    mz[k] = pk::fma(x1[k], zm1, mz[k]);
  };
  auto add_z = [&](int k, const ulonglong2& E, f2 wr, f2 wi, f2 nwr, f2 y, f2 a, f2 b) {
    const f2 ur = pk::fma(E.x, wr, pk::mul(E.y, wi));  // u = conj(E) W
    const f2 ui = pk::fma(E.x, wi, pk::mul(E.y, nwr));
    z[0][0][k] = pk::fma(y, ur, z[0][0][k]);
    z[0][1][k] = pk::fma(y, ui, z[0][1][k]);
    z[1][0][k] = pk::fma(a, ur, z[1][0][k]);
    z[1][1][k] = pk::fma(a, ui, z[1][1][k]);
    z[2][0][k] = pk::fma(b, ur, z[2][0][k]);
    z[2][1][k] = pk::fma(b, ui, z[2][1][k]);
  };
  auto pulse = [&](int i, f2& c, f2& s, f2& ms) {
    const ulonglong2 t0 = *reinterpret_cast<const ulonglong2*>(ctab + i);
    c = t0.x;
    s = t0.y;
    ms = *reinterpret_cast<const f2*>(ntab + i);
  };

  auto sum8 = [](const float* q) {  // the warps' parts of one sum
    const float4 u = reinterpret_cast<const float4*>(q)[0], v = reinterpret_cast<const float4*>(q)[1];
    return ((u.x + u.y) + (u.z + u.w)) + ((v.x + v.y) + (v.z + v.w));
  };
  int buf = 0, par = 0;
  for (int nt = na; nt < ne; nt += kTabs) {
  __syncthreads();  // the previous tables are no longer read
  tables(nt);
  __syncthreads();
  if (live) phases(buf, 0);
  const int nte = min(ne, nt + kTabs);
  for (int n0 = nt; n0 < nte; n0 += CT) {
    const int i0 = n0 - nt;                   // table position
    const float4* E = ering + buf * CT * kWP + lr;
    if (live) {
      // the next chunk's phases go into the buffer of the one before, which every lane has
      // read; then this chunk's have arrived
      __syncwarp();
      if (n0 + CT < nte) {
        phases(buf ^ 1, i0 + CT);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
      } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      }
      __syncwarp();
    }
    if constexpr (MODE == RX_JHW) {
      if (live) {
#pragma unroll
        for (int t = 0; t < CT; ++t) {
          f2 c, s, ms;
          pulse(i0 + t, c, s, ms);
          const float2 w = wtab[(i0 + t) * kTX + lx];
          const f2 wr = pk::both(w.x), wi = pk::both(w.y), nwr = pk::both(-w.x);
#pragma unroll
          for (int k = 0; k < kRP; ++k) {
            const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(E + t * kWP + k * kLR);
            rotate(k, c, s, ms);
            add_z(k, e, wr, wi, nwr, my[k], ay[k], by[k]);
            decay(k);
          }
        }
      }
    } else {
      f2 ys[MODE == RX_JHJV ? CT : 1][3][kRP];
      float acc[2 * CT];
      if (live) {
#pragma unroll
        for (int t = 0; t < CT; ++t) {
          f2 c, s, ms;
          pulse(i0 + t, c, s, ms);
          f2 s1 = 0ull, s2 = 0ull, s3 = 0ull;  // sums of Ex qr, Ey qi, Ex qi + Ey qr
#pragma unroll
          for (int k = 0; k < kRP; ++k) {
            const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(E + t * kWP + k * kLR);
            rotate(k, c, s, ms);
            f2 qr, qi;
            if constexpr (MODE == RX_JHJV) {
              const ulonglong2 q0 = qtab[(3 * k) * kMaxThreads], q1 = qtab[(3 * k + 1) * kMaxThreads], q2 = qtab[(3 * k + 2) * kMaxThreads];
              qr = pk::fma(q1.x, ay[k], pk::fma(q2.x, by[k], pk::mul(q0.x, my[k])));
              qi = pk::fma(q1.y, ay[k], pk::fma(q2.y, by[k], pk::mul(q0.y, my[k])));
            } else {
              qr = pk::mul(qr0[k], my[k]);
              qi = pk::mul(qi0[k], my[k]);
              if (NCH > 1) {
                qr = pk::fma(qr1[k], ay[k], pk::fma(qr2[k], by[k], qr));
                qi = pk::fma(qi1[k], ay[k], pk::fma(qi2[k], by[k], qi));
              }
            }
            s1 = pk::fma(e.x, qr, s1);
            s2 = pk::fma(e.y, qi, s2);
            s3 = pk::fma(e.x, qi, pk::fma(e.y, qr, s3));
            if (MODE == RX_JHJV) {
              ys[t][0][k] = my[k];
              ys[t][1][k] = ay[k];
              ys[t][2][k] = by[k];
            }
            decay(k);
          }
          const float2 a1 = pk::split(s1), a2 = pk::split(s2), a3 = pk::split(s3);
          acc[2 * t] = (a1.x - a2.x) + (a1.y - a2.y);
          acc[2 * t + 1] = a3.x + a3.y;
        }
        // over the warp's eight row lanes by halving: the lanes of a column end with the
        // 2 CT / 8 values of lr (CT = 8: TR lr), or (CT = 2) with value lr / 2 after a last plain
        // sum
#pragma unroll
        for (int n = 2 * CT, off = 16; n > 1 && off >= kTX; n >>= 1, off >>= 1) {
          const bool up = lane & off;
#pragma unroll
          for (int i = 0; i < n / 2; ++i) {
            const float send = up ? acc[i] : acc[i + n / 2], keep = up ? acc[i + n / 2] : acc[i];
            acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
          }
        }
        if (CT == 2) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], kTX);
      } else {
        acc[0] = acc[1] = 0.f;
      }
      float* pb = part + par * NV * kMaxWarps;
      if (CT == 8) {
        pb[((2 * lr) * kTX + lx) * kMaxWarps + warp] = acc[0];
        pb[((2 * lr + 1) * kTX + lx) * kMaxWarps + warp] = acc[1];
      } else if ((lr & 1) == 0) {
        pb[((lr >> 1) * kTX + lx) * kMaxWarps + warp] = acc[0];
      }
      __syncthreads();
      if (MODE == RX_JV) {
        if (warp == (n0 / CT) % W) {
          // lane (t, column): both parts of A[n0 + t][column]
          const int n = n0 + lr;
          const float re = sum8(pb + (2 * lr * kTX + lx) * kMaxWarps);
          const float im = sum8(pb + ((2 * lr + 1) * kTX + lx) * kMaxWarps);
          if (n < ne && ix < nx) P.A[(size_t)n * nx + ix] = make_float2(re, im);
        }
      } else {
        // every warp adds the warps' parts for itself: lane (value, column), then the lanes of
        // a column exchange them
        const float a = sum8(pb + (lane % NV) * kMaxWarps);
        if (live) {
#pragma unroll
          for (int t = 0; t < CT; ++t) {
            const float ar = __shfl_sync(0xffffffffu, a, (2 * t) * kTX + lx);
            const float ai = __shfl_sync(0xffffffffu, a, (2 * t + 1) * kTX + lx);
            const f2 wr = pk::both(ar), wi = pk::both(ai), nwr = pk::both(-ar);
#pragma unroll
            for (int k = 0; k < kRP; ++k) {
              const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(E + t * kWP + k * kLR);
              add_z(k, e, wr, wi, nwr, ys[MODE == RX_JHJV ? t : 0][0][k], ys[MODE == RX_JHJV ? t : 0][1][k],
                    ys[MODE == RX_JHJV ? t : 0][2][k]);
            }
          }
        }
      }
    }
    buf ^= 1;
    par ^= 1;
  }
  }
  if constexpr (MODE != RX_JV) {
  // this segment's gradient: the echo factors, then the inner products with d(rho m)/d alpha
#pragma unroll
  for (int k = 0; k < kRP; ++k) {
    float2 zz[3][2];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      zz[c][0] = pk::split(z[c][0][k]);
      zz[c][1] = pk::split(z[c][1][k]);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const bool o = on[k] && r0[k] + h < ny;
      const int j = o ? (r0[k] + h) * nx + ix : 0;
      const float m = o ? P.maskf[j] * P.scale : 0.f;
      const float2 rh = o ? P.rho[j] : make_float2(0.f, 0.f);
      const float e = o ? P.fac[4 * nvp + ci[k] + h] : 0.f, d = o ? P.fac[5 * nvp + ci[k] + h] : 0.f;
      auto pick = [&](const float2& t) { return h ? t.y : t.x; };
      const float z0r = pick(zz[0][0]), z0i = pick(zz[0][1]);
      const float z1r = e * pick(zz[1][0]), z1i = e * pick(zz[1][1]);
      const float z2r = fmaf(e, pick(zz[2][0]), d * z0r), z2i = fmaf(e, pick(zz[2][1]), d * z0i);
      float* gb = gbuf + (r0[k] + h) * kTX + lx;
      gb[0] = (rh.x * z1i - rh.y * z1r) * m;  // Im(conj(rho) Z1)
      gb[rows * kTX] = (rh.x * z2i - rh.y * z2r) * m;
      gb[2 * rows * kTX] = e * z0i * m;
      gb[3 * rows * kTX] = -e * z0r * m;
    }
  }
  // the blocks of a cluster are the segments of one tile: each adds its share of the elements
  // over all of them (in segment order) from their shared memories
  namespace cgp = cooperative_groups;
  cgp::cluster_group cl = cgp::this_cluster();
  cl.sync();
  const int E = 4 * rows * kTX;
  const int ea = (int)((int64_t)E * sg / P.nseg), ee = (int)((int64_t)E * (sg + 1) / P.nseg);
  // <v, g> and <v, v>: float32 over four elements at most, then float64
  double a = 0.0, b = 0.0;
  float sd = 0.f, sv = 0.f;
  int held = 0;
  for (int e = ea + tid; e < ee; e += nthr) {
    float t = 0.f;
    for (int q = 0; q < P.nseg; ++q) t += cl.map_shared_rank(gbuf, q)[e];
    const int i = e / (rows * kTX), r = e / kTX - i * rows, col = tile * kTX + e % kTX;
    if (r < ny && col < nx) {
      const size_t j = (size_t)i * nv + (size_t)r * nx + col;
      P.g[j] = t;
      if (MODE == RX_JHJV && P.vdot != nullptr) {
        const float vk = P.v[j];
        sd = fmaf(vk, t, sd);
        sv = fmaf(vk, vk, sv);
        if ((++held & 3) == 0) {
          a += (double)sd;
          b += (double)sv;
          sd = sv = 0.f;
        }
      }
    }
  }
  cl.sync();  // no block leaves while its gradient is being read
  if (MODE != RX_JHJV || P.vdot == nullptr) return;
  // <v, g> and <v, v>: this block's parts, then the last block adds all of them in order
  __shared__ double ws[2][kMaxWarps];
  __shared__ int s_last;
  a = red::warp_sum(a + (double)sd);
  b = red::warp_sum(b + (double)sv);
  if (lane == 0) {
    ws[0][warp] = a;
    ws[1][warp] = b;
  }
  __syncthreads();
  if (warp != 0) return;
  const int blocks = gridDim.x;
  if (lane == 0) {
    a = b = 0.0;
    for (int i = 0; i < W; ++i) {
      a += ws[0][i];
      b += ws[1][i];
    }
    P.red[blockIdx.x] = a;
    P.red[blocks + blockIdx.x] = b;
    __threadfence();
    s_last = atomicAdd(P.ticket, 1u) == (unsigned)blocks - 1;
  }
  __syncwarp();
  if (!s_last) return;
  __threadfence();
  a = b = 0.0;
  for (int t = lane; t < blocks; t += 32) {
    a += ((volatile double*)P.red)[t];
    b += ((volatile double*)P.red)[blocks + t];
  }
  a = red::warp_sum(a);
  b = red::warp_sum(b);
  if (lane == 0) {
    *P.vdot = a;
    if (P.vv != nullptr) *P.vv = b;
    *P.ticket = 0u;
  }
  }
}

// One time course channel (0 m_y, 1 and 2 its ln T1 and ln T2 tangents) of one voxel and
// segment per thread, from the kept states into out[n][j] (mrstat_timecourses).
template <int C>
__global__ void __launch_bounds__(128)
rx_timecourse_kernel(const float* __restrict__ fac, const float* __restrict__ st, const float* __restrict__ maskf,
                     const float4* __restrict__ csp, int nx, int nys, int nv, int ntr, int seg, float* __restrict__ out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x, sg = blockIdx.y;
  if (j >= nv) return;
  const size_t nvp = (size_t)nx * nys, e = (size_t)(j % nx) * nys + j / nx;
  const float x1 = fac[e], x2 = fac[nvp + e], d1 = fac[2 * nvp + e], d2 = fac[3 * nvp + e], ee = fac[4 * nvp + e],
              de = fac[5 * nvp + e];
  const float* s0 = st + (size_t)sg * 6 * nvp + e;
  float my = s0[0], mz = s0[nvp], ay = s0[2 * nvp], az = s0[3 * nvp], by = s0[4 * nvp], bz = s0[5 * nvp];
  const float m = maskf[j];
  const int ne = min(ntr, (sg + 1) * seg);
#pragma unroll 4
  for (int n = sg * seg; n < ne; ++n) {
    const float4 cs = __ldg(csp + 2 * n);
    const float c = cs.x, s = cs.z;
    float t = c * my + s * mz;
    mz = c * mz - s * my;
    my = t;
    if (C == 1) {
      t = c * ay + s * az;
      az = c * az - s * ay;
      ay = t;
    }
    if (C == 2) {
      t = c * by + s * bz;
      bz = c * bz - s * by;
      by = t;
    }
    __stcs(out + (size_t)n * nv + j, C == 0 ? m * ee * my : C == 1 ? m * ee * ay : m * fmaf(ee, by, de * my));
    const float zm1 = mz - 1.f;
    if (C == 1) {
      ay = fmaf(x2, ay, ay);
      az = fmaf(x1, az, fmaf(d1, zm1, az));
    }
    if (C == 2) {
      by = fmaf(x2, by, fmaf(d2, my, by));
      bz = fmaf(x1, bz, bz);
    }
    my = fmaf(x2, my, my);
    mz = fmaf(x1, zm1, mz);
  }
}

// One thread per TR and per (ky, row pair); roots[k] = exp(-2 pi i k / ny).
__global__ void __launch_bounds__(256)
rx_tables_kernel(const float2* __restrict__ cs, const float2* __restrict__ roots, int ntr_pad, int ny, int np,
                 float4* __restrict__ csp, float4* __restrict__ etab, unsigned* __restrict__ ticket) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) *ticket = 0u;
  if (i < ntr_pad) {
    const float2 t = cs[i];
    csp[2 * i] = make_float4(t.x, t.x, t.y, t.y);
    csp[2 * i + 1] = make_float4(-t.y, -t.y, 0.f, 0.f);
  }
  if (i < ny * np) {
    const int ky = i / np, iy = 2 * (i - ky * np);
    const float2 zero = make_float2(0.f, 0.f);
    const float2 a = iy < ny ? roots[ky * iy % ny] : zero, b = iy + 1 < ny ? roots[ky * (iy + 1) % ny] : zero;
    etab[i] = make_float4(a.x, b.x, a.y, b.y);
  }
}

template <int NCH, int MODE>
cudaError_t launch_product_t(const Plan& p, RxArgs& a, cudaStream_t st) {
  constexpr int CT = chunk_of(MODE);
  const int W = block_warps(p.ny), threads = 32 * W;
  const size_t sm = sizeof(float4) * W * 2 * CT * kWP + (MODE == RX_JHW ? sizeof(float2) * kTabs * kTX : 0) +
                    kTabs * (sizeof(float4) + sizeof(float2) + sizeof(int)) +
                    (MODE == RX_JHW ? 0 : sizeof(float) * 2 * 2 * CT * kTX * kMaxWarps) +
                    (MODE == RX_JHJV ? sizeof(ulonglong2) * 3 * kRP * kMaxThreads : 0) +
                    (MODE == RX_JV ? 0 : sizeof(float) * 4 * W * kWP * 2 * kTX);
  cudaError_t e =
      cudaFuncSetAttribute(rx_product_kernel<NCH, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.tiles * a.nseg);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;  // the segments of a tile add their gradients
  attr[0].val.clusterDim.x = MODE == RX_JV ? 1 : a.nseg;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, rx_product_kernel<NCH, MODE>, (RxArgs)a);
}

RxArgs args_of(const Plan& p, const RxLin& L, const float2* rho, const float* maskf) {
  RxArgs a = {};
  a.fac = L.fac;
  a.st = L.st;
  a.ns = L.ns;
  a.rho = rho;
  a.maskf = maskf;
  a.csp = p.csp;
  a.kyi = p.kyi;
  a.etab = p.rx_etab;
  a.nx = p.nx;
  a.ny = p.ny;
  a.nys = rx_nys(p);
  a.nv = p.nv;
  a.ntr = p.ntr;
  a.ntr_pad = p.ntr_pad;
  a.seg = L.seg;
  a.nseg = L.nseg;
  a.tiles = (p.nx + kTX - 1) / kTX;
  a.scale = 1.f;
  a.A = p.A;
  a.ticket = p.rx_ticket;
  a.red = p.red;
  a.gate = p.gate;
  return a;
}

}  // namespace

// Whether the plan's exact model runs on this path (the B1 map is a call's argument).
bool rx_supported(const Plan& p) { return p.ny <= kMaxNy && p.npar == 4; }

// The plan's tables for the products, built on the device from its own (on the host, with a
// copy, they were 0.15 ms of a 1.4 ms plan at 224 x 224): the pulses of the TRs, the ticket
// and the phases the products copy, for every ky the (Re, Re, Im, Im) of
// exp(-2 pi i ky iy / ny) for the row pairs (2 p, 2 p + 1), zero past ny.
cudaError_t rx_tables(Plan* p) {
  const int np = block_warps(p->ny) * kWP;
  const size_t npulse = 2 * (size_t)p->ntr_pad, nphase = (size_t)p->ny * np;
  cudaError_t e = dalloc(p, &p->rx_tab, npulse + nphase + 1);
  if (e != cudaSuccess) return e;
  p->csp = p->rx_tab;
  p->rx_etab = p->rx_tab + npulse;
  p->rx_ticket = reinterpret_cast<unsigned*>(p->rx_tab + npulse + nphase);
  const int n = std::max(p->ntr_pad, (int)nphase);
  rx_tables_kernel<<<(n + 255) / 256, 256>>>(p->cs, p->roots, p->ntr_pad, p->ny, np, p->csp, p->rx_etab, p->rx_ticket);
  return cudaGetLastError();
}

// TRs per segment (a multiple of 8): the number of segments that balances the blocks
// (column tiles x segments) over the SMs.  A block costs its TRs plus a prologue worth about
// a dozen TRs (loads of factors, states and coefficients) and the SMs run two blocks of up
// to 256 threads each, more of the smaller ones; at least 16 TRs per segment, and at most
// eight segments (the largest portable cluster).
int rx_segment(const Plan& p, int sms) {
  const int tiles = (p.nx + kTX - 1) / kTX, threads = 32 * block_warps(p.ny);
  const int64_t slots = (int64_t)sms * std::max(2, std::min(16, 2 * kMaxThreads / threads));
  int best = (p.ntr + 7) / 8 * 8;
  int64_t cost = INT64_MAX;
  for (int n = 1; n <= std::max(1, std::min(kMaxSegments, p.ntr / 16)); ++n) {
    const int seg = ((p.ntr + n - 1) / n + 7) / 8 * 8;
    const int64_t blocks = (int64_t)tiles * ((p.ntr + seg - 1) / seg);
    const int64_t c = (blocks + slots - 1) / slots * (seg + 12);
    if (c < cost) {
      cost = c;
      best = seg;
    }
  }
  return best;
}

// Linearisation at alpha into L (allocated; L.ns 6 with the tangents, 2 for m alone): rho
// (masked) and, where given, the mask as floats.
cudaError_t launch_rx_states(const Plan& p, const RxLin& L, const float* alpha, const uint8_t* mask, float2* rho,
                             float* maskf, cudaStream_t st) {
  const int nys = rx_nys(p);
  const int blocks = (int)(((int64_t)p.nx * nys + 127) / 128);
  const float te = (float)p.te_ms, tr = (float)p.tr_ms, m0z = p.inversion ? -1.f : 1.f;
  auto kernel = L.ns == 2 ? rx_states_kernel<1> : rx_states_kernel<3>;
  kernel<<<blocks, 128, 0, st>>>(alpha, mask, p.cs, p.nx, p.ny, nys, p.nv, p.ntr, L.seg, L.nseg, te, tr, m0z, L.fac,
                                 L.st, rho, maskf);
  return cudaGetLastError();
}

// Phase-encode sums of the signal into p.A (never gated)
cudaError_t launch_rx_signal(const Plan& p, const RxLin& L, const float2* rho, cudaStream_t st) {
  RxArgs a = args_of(p, L, rho, nullptr);
  a.gate = nullptr;
  return launch_product_t<1, RX_JV>(p, a, st);
}

// Phase-encode sums of J.v into p.A
cudaError_t launch_rx_jv(const Plan& p, const RxLin& L, const float* v, cudaStream_t st) {
  RxArgs a = args_of(p, L, p.rho, p.maskf);
  a.v = v;
  return launch_product_t<3, RX_JV>(p, a, st);
}

cudaError_t launch_rx_jhw(const Plan& p, const RxLin& L, const float2* rho, const float* maskf, const float2* wt,
                          float* g, cudaStream_t st) {
  RxArgs a = args_of(p, L, rho, maskf);
  a.wt = wt;
  a.g = g;
  return launch_product_t<3, RX_JHW>(p, a, st);
}

// Re(J^H J) v for nkx == nx; with vdot also <v, g> and (with vv) <v, v>
cudaError_t launch_rx_jhjv(const Plan& p, const RxLin& L, const float* v, float* g, double* vdot, double* vv,
                           cudaStream_t st) {
  RxArgs a = args_of(p, L, p.rho, p.maskf);
  a.v = v;
  a.g = g;
  a.scale = (float)p.nx;
  a.vdot = vdot;
  a.vv = vv;
  return launch_product_t<3, RX_JHJV>(p, a, st);
}

cudaError_t launch_rx_timecourse(const Plan& p, const RxLin& L, int channel, float* out, cudaStream_t st) {
  if (p.nv == 0) return cudaSuccess;
  const dim3 grid((p.nv + 127) / 128, L.nseg);
  auto kernel = channel == 0 ? rx_timecourse_kernel<0> : channel == 1 ? rx_timecourse_kernel<1> : rx_timecourse_kernel<2>;
  kernel<<<grid, 128, 0, st>>>(L.fac, L.st, p.maskf, p.csp, p.nx, rx_nys(p), p.nv, p.ntr, L.seg, out);
  return cudaGetLastError();
}

}  // namespace mrstat
