// kinetic.cu -- the mesoscopic kinetic step of GSIS on sm_103a (Section 3.2 of arXiv 2310.18916).
//
// One CTA owns one block of VB = 32 discrete velocities of a single octant (one per lane) and
// marches through the spatial cells colour by colour, the colours being the hyperplanes
// i' + j' + k' = const in the upwind order of that octant.  For each cell and velocity it
//   - applies the pending VDF correction of Eq. updatef (and the closed-domain mass scale)
//     while staging f^n into a three-colour shared-memory ring,
//   - builds the reference distribution g (Shakhov g_0t, Section 2.2),
//   - takes the LSQ gradient and the Venkatakrishnan limiter, reconstructs the outflow face
//     value (second-order upwind, Section 3.2),
//   - solves the point-implicit delta form with the first-order upwind implicit operator,
//     taking the inflow value "face value + upwind increment" from the previous colour
//     (exact in one pass on a rectilinear grid: every inflow neighbour has a lower colour),
//   - writes f^{n+1/2} in place, and the outgoing flux moments of its wall faces.
// The velocity moments of f^{n+1/2} are a separate streaming pass (moments_kernel, and
// moments_origin_kernel for FP64 storage on tensor-product grids).
#include <algorithm>

#include "kinetic_device.cuh"

namespace gsis {

// ---- bulk asynchronous copies (TMA) into shared memory, completed on an mbarrier ----
__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// the one arrival of a phase, announcing the bytes its copies will deliver
__device__ __forceinline__ void mbar_expect(uint64_t *bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_test(uint64_t *bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// bounded wait for the phase of the given parity; false on time-out (about a second)
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned parity, long long limit = 1LL << 31) {
  const long long t0 = clock64();
  for (unsigned i = 0; !mbar_test(bar, parity); ++i)
    if ((i & 63u) == 63u && clock64() - t0 > limit) return false;
  return true;
}

// Self-test of the bounded mbarrier wait: a phase that no arrival and no copy completes, so the
// wait runs out after `limit` cycles and raises GSIS_ERR_TIMEOUT.
__global__ void mbarrier_timeout_probe(int *err, long long limit) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) mbar_init(&bar);
  __syncthreads();
  const bool ok = mbar_wait(&bar, 0u, limit);
  if (!ok && threadIdx.x == 0) atomicCAS(err, 0, GSIS_ERR_TIMEOUT);
}

cudaError_t probe_mbarrier_timeout(int *err, long long limit, cudaStream_t s) {
  mbarrier_timeout_probe<<<1, 32, 0, s>>>(err, limit);
  return cudaGetLastError();
}

// global -> shared bulk copy of `bytes` (a multiple of 16, both addresses 16-byte aligned)
__device__ __forceinline__ void bulk_copy(void *dst, const void *src, unsigned bytes, uint64_t *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}

template <typename T>
__device__ __forceinline__ void load_state_shared(const T *src, T *st, int n) {
#pragma unroll
  for (int q = 0; q < 40; ++q)
    if (q < n) st[q] = src[q];
}

// memory layout of the kinetic kernel: the ring of three colours (four in global memory) and the
// face buffers (T), the bulk-copy staging area for one colour (stored f in S, then the state rows
// in T), the mbarrier and the time-out flag
__host__ __device__ constexpr int ring_slots(bool gm) { return gm ? 4 : 3; }
template <typename T, typename S>
struct KinSmem {
  size_t ring, ebuf, rawf, rawst, bar, total;
  __host__ __device__ KinSmem(const KinGeom &g, int nv, int sl, bool gm) {
    ring = 0;
    ebuf = ring + (size_t)ring_slots(gm) * g.maxcol * nv * VB * sizeof(T);
    rawf = ebuf;
    for (int a = 0; a < 3; ++a) rawf += (size_t)g.ntrans[a] * nv * VB * sizeof(T);
    rawf = (rawf + 15) & ~(size_t)15;
    rawst = (rawf + (size_t)g.maxcol * nv * VB * sizeof(S) + 15) & ~(size_t)15;
    bar = (rawst + (size_t)g.maxcol * sl * sizeof(T) + 15) & ~(size_t)15;
    total = bar + 16;
  }
};

// FX: factored Maxwellians (FP64 on a tensor-product velocity grid).  An FP64 exponential is many
// instructions of a pipe that retires one warp instruction in 19 cycles per SM, but on a product
// grid exp(-|xi - u|^2 / T) is the product of three one-dimensional factors, and the polynomials in
// c = xi - u of the reference distributions are sums of three.  factor_table_kernel writes per cell
// and grid node of each axis (32 times fewer than points):
//   Shakhov  {e_n, e_o, p, s}: the factors of M(W^n) and M(W^{n-1/2}) (the x ones with the constant
//            in front), p = A q_a c_a and s = c_a^2 / T_t (the z one less 5/2), so that
//            g = M (1 + sum p sum s);
//   Rykov    {e_n, e_o, e_T, c_a^2, A q_a c_a, and the coefficients of c_a in g_r, g_1t, g_1r}.
// With one limiter evaluation per cell (see venkat_parts) and signs and bounds kept on the integer
// pipe the 2D Shakhov step takes about 56 FP64 instructions per point instead of 118, 85 % of the
// FP64 pipe's rate: 128^2 cells with 32^3 velocities 115.1 -> 62.7 ms (floor of those instructions
// 57), the wall pre-pass 4.2 -> 1.1; Rykov 48^2 with 20^3 10.9 -> 5.2.  FP32 keeps its exponentials
// (MUFU), cheaper there than gathered factors.

__global__ void __launch_bounds__(128) factor_table_kernel(int nc, int nx, int ny, int nz, int nvdf, const double *st64,
                                                           const double *vaxis, double *tab) {
  const int nn = nx + ny + nz;
  const size_t n = (size_t)nc * nn;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int node = (int)(i % nn);
    const size_t cell = i / nn;
    const int a = node < nx ? 0 : (node < nx + ny ? 1 : 2);
    const double *st = st64 + cell * NST;
    const double xi = vaxis[node], c = xi - st[a], co = xi - st[5 + a];
    double *o = tab + i * factor_table_len(nvdf);
    double en = exp(-c * c * st[3]), eo = exp(-co * co * st[8]);
    if (a == 0) {
      en *= st[4];
      eo *= st[9];
    }
    o[0] = en;
    o[1] = eo;
    if (nvdf == 1) {
      o[2] = st[12 + a] * c;
      o[3] = c * c * st[3] - (a == 2 ? 2.5 : 0.0);
    } else {
      o[2] = exp(-c * c * st[24]) * (a == 0 ? st[25] : 1.0);
      o[3] = c * c;
      o[4] = st[12 + a] * c;
      o[5] = st[26 + a] * c;
      o[6] = st[31 + a] * c / st[4];
      o[7] = st[34 + a] * c / st[25];
    }
  }
}

cudaError_t launch_factor_table(int nc, const int *nv_axis, int nvdf, const double *st64, const double *vaxis, double *tab,
                                cudaStream_t s) {
  const size_t n = (size_t)nc * (nv_axis[0] + nv_axis[1] + nv_axis[2]);
  const size_t grid = std::min<size_t>((n + 127) / 128, 152 * 16);
  factor_table_kernel<<<(unsigned)grid, 128, 0, s>>>(nc, nv_axis[0], nv_axis[1], nv_axis[2], nvdf, st64, vaxis, tab);
  return cudaGetLastError();
}

// f^n of the NV reduced VDFs from the cell's factor rows of this lane's three nodes (Eq. updatef)
template <int NV>
__device__ __forceinline__ void corrected_factored(const double *stored, const double *row, const int *node, double s,
                                                   double cn, double co, double *f) {
  constexpr int L = factor_table_len(NV);
  double2 e[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) e[a] = __ldg(reinterpret_cast<const double2 *>(row + node[a] * L));
  const double tn = e[0].x * e[1].x, to = e[0].y * e[1].y;
  if constexpr (NV == 1) {
    f[0] = fma(tn, e[2].x, fma(-to, e[2].y, s * stored[0]));
  } else {
    // f1 carries the internal-energy factors cn, co of the two Maxwellians
    const double mn = tn * e[2].x, mo = to * e[2].y;
    f[0] = fma(s, stored[0], mn - mo);
    f[1] = fma(s, stored[1], fma(cn, mn, -co * mo));
  }
}

// GM: the colour ring and face buffers of a velocity block too large for shared memory (3D
// meshes: a colour of n^3 cells has O(n^2) cells) live in the block's own slice of a global
// scratch (L2-resident where it fits), and each colour is staged with plain loads.  The
// arithmetic and the order of every cell's inputs are those of the shared-memory kernel.
template <typename T, typename S, int NACT, int NV, bool GM, bool FX>
__global__ void kinetic_kernel(const KinArgs<T, S> A) {
  extern __shared__ __align__(16) unsigned char smem_dyn[];
  const KinGeom &G = A.g;
  constexpr int SL = stage_state_len<S, NV>();
  const KinSmem<T, S> L(G, NV, SL, GM);
  unsigned char *smem_raw = GM ? A.gscratch + (size_t)blockIdx.x * A.gstride : smem_dyn;
  T *ring = reinterpret_cast<T *>(smem_raw + L.ring);
  T *ebuf[3];
  {
    T *p = reinterpret_cast<T *>(smem_raw + L.ebuf);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      ebuf[a] = p;
      p += (size_t)G.ntrans[a] * NV * VB;
    }
  }
  S *rawf = reinterpret_cast<S *>(smem_raw + L.rawf);
  T *rawst = reinterpret_cast<T *>(smem_raw + L.rawst);
  uint64_t *bar = reinterpret_cast<uint64_t *>(smem_raw + L.bar);
  volatile int *dead = reinterpret_cast<volatile int *>(smem_raw + L.bar + 8);  // a wait for copies timed out
  const int b = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int oct = A.boct[b];
  const int sg[3] = {oct & 1 ? -1 : 1, oct & 2 ? -1 : 1, oct & 4 ? -1 : 1};
  const T *vp = A.vel + ((size_t)b * VB + lane) * 4;
  const T xi[3] = {vp[0], vp[1], vp[2]};
  const T wv = vp[3];
  // factored Maxwellians: this lane's nodes in a cell's rows
  int node[3] = {0, 0, 0};
  if constexpr (FX) {
    const int packed = A.vnode[(size_t)b * VB + lane];
    node[0] = packed & 1023;
    node[1] = packed >> 10 & 1023;
    node[2] = packed >> 20;
  }
  const unsigned frow = A.nnode * factor_table_len(NV);  // doubles per cell of the table
  const T e2 = (T)0.5 * (xi[0] * xi[0] + xi[1] * xi[1] + xi[2] * xi[2]);
  T axi[3], Mw[3], Mw1[3];
  int upside[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    axi[a] = fabs(xi[a]);
    upside[a] = 2 * a + (sg[a] > 0 ? 0 : 1);
    Mw[a] = Mw1[a] = (T)0;
    if (a < NACT && G.wall_base[upside[a]] >= 0) {
      Mw[a] = wall_maxwellian<T>(A.wall_uT + 4 * upside[a], xi[0], xi[1], xi[2]);
      // re-emitted f1 = (d_r T_w / 4) f0 at the wall
      if constexpr (NV == 2) Mw1[a] = (T)(A.d_r * A.wall_uT[4 * upside[a] + 3] / 4.0) * Mw[a];
    }
  }
  const int n0 = G.n[0], n1 = G.n[1];
  S *F[NV];
  F[0] = A.f + (size_t)b * G.nc * VB;
  if constexpr (NV == 2) F[NV - 1] = A.f1 + (size_t)b * G.nc * VB;
  const int4 *natcell = A.natcell + (size_t)oct * G.nc;
  const size_t slot_stride = (size_t)G.maxcol * NV * VB;
  const int tid = threadIdx.x, nthr = blockDim.x;
  // Colour c + 2's stored f rows (VB values per cell and VDF) and state rows are copied into the
  // staging area by bulk copies while colour c is computed; one thread per copy, the cell index
  // loaded before the wait so that its latency is hidden.
  constexpr unsigned kRowBytes = VB * sizeof(S), kStBytes = SL * sizeof(T);
  auto colour_bytes = [&](int c) { return (unsigned)(A.col_off[c + 1] - A.col_off[c]) * (NV * kRowBytes + kStBytes); };
  auto prefetch_cell = [&](int c) {
    if (c >= G.ncol) return 0;
    const int off = A.col_off[c], cnt = A.col_off[c + 1] - off;
    return tid < cnt * (NV + 1) ? __ldg(&natcell[off + tid / (NV + 1)].x) : 0;
  };
  auto issue = [&](int c, int cell0) {
    const int off = A.col_off[c], cnt = A.col_off[c + 1] - off;
    for (int i = tid; i < cnt * (NV + 1); i += nthr) {
      const int p = i / (NV + 1), q = i - p * (NV + 1);
      const int cell = i == tid ? cell0 : __ldg(&natcell[off + p].x);
      if (q < NV)
        bulk_copy(rawf + (size_t)(p * NV + q) * VB, F[q] + (size_t)cell * VB, kRowBytes, bar);
      else
        bulk_copy(rawst + (size_t)p * SL, state_of(A.st, cell), kStBytes, bar);
    }
  };
  // Each colour is one phase of the mbarrier, waited for by every thread; on a time-out the thread
  // flags the error, and the block leaves at its next barrier after another (bounded) wait for its
  // copies in flight.
  unsigned phase = 0;
  auto await = [&]() {
    if (!mbar_wait(bar, phase & 1u)) {
      atomicCAS(A.err, 0, GSIS_ERR_TIMEOUT);
      *dead = 1;
    }
    ++phase;
  };
  constexpr int NS = ring_slots(GM);
  auto stage = [&](int c) {
    const int off = A.col_off[c], cnt = A.col_off[c + 1] - off;
    T *slot = ring + (size_t)(c % NS) * slot_stride;
    for (int p = warp; p < cnt; p += nw) {
      T st[SL], stored[NV], f[NV];
      if constexpr (GM) {
        const int cell = __ldg(&natcell[off + p].x);
        load_state<SL>(state_of(A.st, cell), st);
#pragma unroll
        for (int q = 0; q < NV; ++q) stored[q] = Fio<T, S>::ld(F[q] + (size_t)cell * VB + lane);
      } else {
        load_state_shared<T>(rawst + (size_t)p * SL, st, SL);
#pragma unroll
        for (int q = 0; q < NV; ++q) stored[q] = Fio<T, S>::ld(rawf + (size_t)(p * NV + q) * VB + lane);
      }
      if constexpr (FX) {
        const int cell = __ldg(&natcell[off + p].x);
        corrected_factored<NV>(stored, A.ftab + (size_t)(unsigned)cell * frow, node, st[10], NV == 2 ? st[SL > 29 ? 29 : 0] : 0.0,
                               NV == 2 ? st[SL > 39 ? 39 : 0] : 0.0, f);
      } else {
        corrected_all<T, S, NV>(stored, st, xi[0], xi[1], xi[2], f);
      }
#pragma unroll
      for (int q = 0; q < NV; ++q) slot[(p * NV + q) * VB + lane] = f[q];
    }
  };

  // Global ring: colour c + 2 is staged while colour c is computed, one barrier per colour.  Shared
  // ring: the copies of colour c + 2 run while colour c is computed; colour c + 1 is staged
  // before it.
  if constexpr (GM) {
    stage(0);
    if (G.ncol > 1) stage(1);
    __syncthreads();
  } else {
    if (tid == 0) {
      *dead = 0;
      mbar_init(bar);
      mbar_expect(bar, colour_bytes(0));
    }
    __syncthreads();
    issue(0, prefetch_cell(0));
    const int pf = prefetch_cell(1);
    await();
    stage(0);
    if (tid == 0 && G.ncol > 1) mbar_expect(bar, colour_bytes(1));
    __syncthreads();
    if (*dead) {
      mbar_wait(bar, 0u);
      return;
    }
    if (G.ncol > 1) issue(1, pf);
  }
  for (int c = 0; c < G.ncol; ++c) {
    if constexpr (GM) {
      if (c + 2 < G.ncol) stage(c + 2);
    } else {
      const int pf = prefetch_cell(c + 2);
      if (c + 1 < G.ncol) {
        await();
        stage(c + 1);
        if (tid == 0 && c + 2 < G.ncol) mbar_expect(bar, colour_bytes(c + 2));
      }
      __syncthreads();
      if (*dead) {
        // (the copies awaited in vain may still land: one more bounded wait before the memory goes)
        mbar_wait(bar, (phase - 1) & 1u);
        return;
      }
      if (c + 2 < G.ncol) issue(c + 2, pf);
    }
    const T *slotm = ring + (size_t)((c + NS - 1) % NS) * slot_stride;
    const T *slot0 = ring + (size_t)(c % NS) * slot_stride;
    const T *slotp = ring + (size_t)((c + 1) % NS) * slot_stride;
    const int off = A.col_off[c], cnt = A.col_off[c + 1] - off;
    for (int p = warp; p < cnt; p += nw) {
      const int4 nc4 = __ldg(&natcell[off + p]);
      const int cell = nc4.x;
      const int nat[3] = {nc4.y, nc4.z, nc4.w};
      const EntryInfo &E = entry_of(A.entry, off + p);
      int nb[6], trn[3];
#pragma unroll
      for (int q = 0; q < 2 * NACT; ++q) nb[q] = __ldg(&E.nb[q]);
#pragma unroll
      for (int q = 0; q < NACT; ++q) trn[q] = __ldg(&E.trn[q]);
      T fi[NV];
#pragma unroll
      for (int q = 0; q < NV; ++q) fi[q] = slot0[(p * NV + q) * VB + lane];
      constexpr int CL = NV == 2 ? NST_RYKOV : 16;
      T st[CL];
      load_state<CL>(state_of(A.st, cell), st);
      // gradient (LSQ, decoupled per axis on a rectilinear grid) and the limiter's bounds per VDF, the
      // outflow faces' increments (|r| is the same on both faces of an axis)
      T dout[NV][3], invh[3];
      Largest<T> d2[NV], dp[NV], dn[NV];
#pragma unroll
      for (int a = 0; a < NACT; ++a) {
        const AxisFlow<T> gc = A.flow[a][2 * nat[a] + (sg[a] > 0 ? 0 : 1)];
#pragma unroll
        for (int q = 0; q < NV; ++q) {
          T fup = fi[q], fdn = fi[q];
          if (nb[2 * a] >= 0) fup = slotm[(nb[2 * a] * NV + q) * VB + lane];
          if (nb[2 * a + 1] >= 0) fdn = slotp[(nb[2 * a + 1] * NV + q) * VB + lane];
          const T du = fup - fi[q], dd = fdn - fi[q];
          dp[q].raise(du);
          dp[q].raise(dd);
          dn[q].raise_neg(du);
          dn[q].raise_neg(dd);
          dout[q][a] = gc.up * du + gc.dn * dd;
          d2[q].raise_abs(dout[q][a]);
        }
        invh[a] = gc.invh;
      }
      // the implicit diagonal D = 1/dt + 1/tau + the outflow coefficients, then the limiter.  In
      // FP64 one reciprocal r = 1 / (bd D) gives both phi = bn / bd = bn D r and the update's
      // 1 / D = bd r (bd >= eps^2, which the host keeps far above the smallest normal number)
      T D = st[15];
#pragma unroll
      for (int a = 0; a < NACT; ++a) D += axi[a] * invh[a];
      const T eps2 = __ldg(A.eps2 + cell);
      T phi[NV], invD[NV];
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        if constexpr (std::is_same<T, double>::value) {
          T bn, bd;
          venkat_parts<T>(dp[q], dn[q], d2[q], eps2, bn, bd);
          const T r = rcp_newton(bd * D);
          phi[q] = bn * D * r;
          invD[q] = bd * r;
        } else {
          phi[q] = venkat_phi<T>(dp[q], dn[q], d2[q], eps2);
          invD[q] = (T)0;
        }
      }
      // reference distributions of the state W^n
      T mw, g[NV];  // mw: Maxwellian of W^n
      if constexpr (FX) {
        const T *row = A.ftab + (size_t)(unsigned)cell * frow;
        constexpr int FL = factor_table_len(NV);
        T v[3][FL];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
          for (int t = 0; t < FL; t += 2) {
            const double2 u = __ldg(reinterpret_cast<const double2 *>(row + node[a] * FL + t));
            v[a][t] = u.x;
            v[a][t + 1] = u.y;
          }
        mw = v[0][0] * v[1][0] * v[2][0];
        if constexpr (NV == 1) {
          g[0] = mw * ((v[0][2] + v[1][2] + v[2][2]) * (v[0][3] + v[1][3] + v[2][3]) + (T)1);
        } else {
          const T mT = v[0][2] * v[1][2] * v[2][2], c2 = v[0][3] + v[1][3] + v[2][3];
          const T g0t = mw * ((v[0][4] + v[1][4] + v[2][4]) * (c2 * st[3] - (T)2.5) + (T)1);
          const T g0r = mT * ((v[0][5] + v[1][5] + v[2][5]) * (c2 * st[24] - (T)2.5) + (T)1);
          const T g1t = st[29] * g0t + (v[0][6] + v[1][6] + v[2][6]) * mw;
          const T g1r = st[30] * g0r + (v[0][7] + v[1][7] + v[2][7]) * mT;
          g[0] = st[37] * g0t + st[38] * g0r;
          g[1] = st[37] * g1t + st[38] * g1r;
        }
      } else {
        const T cx = xi[0] - st[0], cy = xi[1] - st[1], cz = xi[2] - st[2];
        reference<T, NV>(st, cx, cy, cz, cx * cx + cy * cy + cz * cz, mw, g);
      }
      T acc[NV];
#pragma unroll
      for (int q = 0; q < NV; ++q) acc[q] = (g[q] - fi[q]) * st[11];
      T fout[NV][3];
#pragma unroll
      for (int a = 0; a < NACT; ++a) {
        const T k = axi[a] * invh[a];
        T rho_w = (T)0;
        if (nb[2 * a] < 0) {
          // upwind boundary: the natural transverse index of the wall face
          const int trw = a == 0 ? nat[1] + n1 * nat[2] : (a == 1 ? nat[0] + n0 * nat[2] : nat[0] + n0 * nat[1]);
          rho_w = (T)A.rho_w[G.wall_base[upside[a]] + trw];
        }
#pragma unroll
        for (int q = 0; q < NV; ++q) {
          fout[q][a] = fi[q] + phi[q] * dout[q][a];
          const T ein = nb[2 * a] >= 0 ? ebuf[a][(trn[a] * NV + q) * VB + lane] : rho_w * (q == 0 ? Mw[a] : Mw1[a]);
          acc[q] -= k * (fout[q][a] - ein);
        }
      }
      T df[NV];
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        if constexpr (std::is_same<T, double>::value) df[q] = acc[q] * invD[q];
        else df[q] = ddiv(acc[q], D);
        // relative storage keeps the deviation from the reference: M_t for f0, (d_r Tr_n / 4) M_t for f1
        const T ref = q == 0 ? mw : st[NV == 2 ? 29 : 0] * mw;
        Fio<T, S>::st(F[q] + (size_t)cell * VB + lane, StoredRelative<S>::value ? fi[q] + df[q] - ref : fi[q] + df[q]);
      }
#pragma unroll
      for (int a = 0; a < NACT; ++a) {
        T eout[NV];
#pragma unroll
        for (int q = 0; q < NV; ++q) {
          eout[q] = fout[q][a] + df[q];
          ebuf[a][(trn[a] * NV + q) * VB + lane] = eout[q];
        }
        if (nb[2 * a + 1] < 0) {
          // outflow face on the domain boundary (a wall): moments of the flux towards the wall
          const int trw = a == 0 ? nat[1] + n1 * nat[2] : (a == 1 ? nat[0] + n0 * nat[2] : nat[0] + n0 * nat[1]);
          const int wid = G.wall_base[2 * a + (sg[a] > 0 ? 1 : 0)] + trw;
          const T fl = wv * xi[a] * eout[0];
          const T e1 = NV == 2 ? wv * xi[a] * eout[NV - 1] : (T)0;
          const T m0 = warp_sum(fl), m1 = warp_sum(fl * xi[0]), m2 = warp_sum(fl * xi[1]);
          const T m3 = warp_sum(fl * xi[2]), m4 = warp_sum(fl * e2 + e1);
          const T m5 = NV == 2 ? warp_sum(e1) : (T)0;
          if (lane == 0) {
            T *W = A.wpart + ((size_t)b * A.nwall + wid) * NWF;
            W[0] = m0;
            W[1] = m1;
            W[2] = m2;
            W[3] = m3;
            W[4] = m4;
            W[5] = m5;
          }
        }
      }
    }
    __syncthreads();
  }
}

template <typename T, typename S>
size_t kinetic_smem_bytes(const KinGeom &g, int nvdf) {
  const int sl = nvdf == 2 ? stage_state_len<S, 2>() : stage_state_len<S, 1>();
  return KinSmem<T, S>(g, nvdf, sl, false).total;
}

// the ring and face buffers only (the bulk-copy staging area is not used from global memory),
// rounded to 256 bytes so that every block's slice starts on an aligned boundary
template <typename T, typename S>
size_t kinetic_gscratch_stride(const KinGeom &g, int nvdf) {
  const int sl = nvdf == 2 ? stage_state_len<S, 2>() : stage_state_len<S, 1>();
  return (KinSmem<T, S>(g, nvdf, sl, true).rawf + 255) & ~(size_t)255;
}

template <typename T, typename S, int NV, bool GM, bool FX>
static void (*kinetic_fn_fx(int nact))(const KinArgs<T, S>) {
  return nact == 1 ? kinetic_kernel<T, S, 1, NV, GM, FX>
                   : (nact == 2 ? kinetic_kernel<T, S, 2, NV, GM, FX> : kinetic_kernel<T, S, 3, NV, GM, FX>);
}

template <typename T, typename S, bool GM>
static void (*kinetic_fn_gm(int nact, int nvdf, bool fx))(const KinArgs<T, S>) {
  if constexpr (std::is_same<T, double>::value)
    if (fx) return nvdf == 2 ? kinetic_fn_fx<T, S, 2, GM, true>(nact) : kinetic_fn_fx<T, S, 1, GM, true>(nact);
  return nvdf == 2 ? kinetic_fn_fx<T, S, 2, GM, false>(nact) : kinetic_fn_fx<T, S, 1, GM, false>(nact);
}

// gm: ring in global scratch; fx: factored Maxwellians
template <typename T, typename S>
static void (*kinetic_fn(const KinGeom &g, int nvdf, bool gm, bool fx))(const KinArgs<T, S>) {
  return gm ? kinetic_fn_gm<T, S, true>(g.nact, nvdf, fx) : kinetic_fn_gm<T, S, false>(g.nact, nvdf, fx);
}

template <typename T, typename S>
cudaError_t kinetic_shape(const KinGeom &g, int nvdf, bool gm, bool fx, int want_warps, size_t smem, int *warps,
                          int *ctas_per_sm) {
  void (*k)(const KinArgs<T, S>) = kinetic_fn<T, S>(g, nvdf, gm, fx);
  cudaFuncAttributes attr;
  cudaError_t e = cudaFuncGetAttributes(&attr, k);
  if (e != cudaSuccess) return e;
  *warps = std::max(1, std::min(want_warps, attr.maxThreadsPerBlock / 32));
  // the limit belongs to the kernel and all host threads' solvers launch it: always what the device
  // allows, never what one solver needs
  int dev = 0, optin = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)attr.sharedSizeBytes);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, k, *warps * 32, smem);
}

template <typename T, typename S>
cudaError_t launch_kinetic(const KinArgs<T, S> &a, int nblocks, int nwarps, size_t smem, cudaStream_t s) {
  void (*k)(const KinArgs<T, S>) = kinetic_fn<T, S>(a.g, a.nvdf, a.gscratch != nullptr, a.ftab != nullptr);
  k<<<nblocks, nwarps * 32, smem, s>>>(a);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Diffuse-wall pre-pass: rho_w of each wall face balances the mass flux of the molecules that
// reach the wall, whose face values are the wall cell's limited reconstruction of f^n.

template <typename T, typename S, int NACT, bool FX>
__global__ void wall_prepass_kernel(const KinArgs<T, S> A, const int *wall_cell, const int *wall_side,
                                    const double *Z0, double *rho_w, int nslots) {
  const KinGeom &G = A.g;
  const int wf = blockIdx.x;
  const int cell = wall_cell[wf], side = wall_side[wf], axn = side / 2;
  const double dir = (side & 1) ? 1.0 : -1.0;
  const int n0 = G.n[0], n1 = G.n[1];
  const int nat[3] = {cell % n0, (cell / n0) % n1, cell / (n0 * n1)};
  const int stride[3] = {1, n0, n0 * n1};
  constexpr int SL = state_len<S>();
  // state rows of the cell and its neighbours (FX: the mass scale only, one for all cells)
  T st[FX ? 1 : SL], stn[FX ? 1 : 3][2][FX ? 1 : SL];
  bool has[3][2];
  if constexpr (FX) st[0] = A.st[(size_t)cell * NST + 10];
  else load_state<SL>(A.st + (size_t)cell * NST, st);
#pragma unroll
  for (int a = 0; a < NACT; ++a) {
    has[a][0] = nat[a] > 0;
    has[a][1] = nat[a] < G.n[a] - 1;
    if constexpr (!FX) {
      if (has[a][0]) load_state<SL>(A.st + (size_t)(cell - stride[a]) * NST, stn[a][0]);
      if (has[a][1]) load_state<SL>(A.st + (size_t)(cell + stride[a]) * NST, stn[a][1]);
    }
  }
  AxisCell<T> gc[3];
#pragma unroll
  for (int a = 0; a < NACT; ++a) gc[a] = A.ax[a][nat[a]];
  const T eps2 = A.eps2[cell];
  // f^n of this thread's velocity in a cell (f0: the mass flux needs no other)
  const unsigned frow = A.nnode * factor_table_len(A.nvdf);
  auto value = [&](int c, const T *sc, size_t at, const T *v, const int *node) {
    const T raw = Fio<T, S>::ld(A.f + at);
    if constexpr (FX) {
      const T *row = A.ftab + (size_t)(unsigned)c * frow;
      const int L = factor_table_len(A.nvdf);
      double2 e[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) e[a] = __ldg(reinterpret_cast<const double2 *>(row + node[a] * L));
      return fma(e[0].x * e[1].x, e[2].x, fma(-(e[0].y * e[1].y), e[2].y, st[0] * raw));
    } else {
      return corrected_stored<T, S>(raw, sc, v[0], v[1], v[2]);
    }
  };
  double acc = 0.0;
  for (int v = threadIdx.x; v < nslots; v += blockDim.x) {
    const T *vp = A.vel + (size_t)v * 4;
    const T xi[3] = {vp[0], vp[1], vp[2]}, w = vp[3];
    const T xa = axn == 0 ? xi[0] : (axn == 1 ? xi[1] : xi[2]);
    // (the direction test and the product in the arithmetic type: FP64 conversions, compares
    // and products per velocity would run at the FP64 rate; dir = +-1 keeps them exact)
    if (!is_positive(w) || !is_positive(xa * (T)dir)) continue;
    const int blk = v / VB, ln = v % VB;
    const size_t base = (size_t)blk * G.nc * VB + ln;
    int node[3] = {0, 0, 0};
    if constexpr (FX) {
      const int packed = A.vnode[v];
      node[0] = packed & 1023;
      node[1] = packed >> 10 & 1023;
      node[2] = packed >> 20;
    }
    const T fi = value(cell, st, base + (size_t)cell * VB, xi, node);
    T dout = (T)0;
    Largest<T> d2, dp, dn;
#pragma unroll
    for (int a = 0; a < NACT; ++a) {
      T dlo = (T)0, dhi = (T)0;
      if (has[a][0]) dlo = value(cell - stride[a], stn[FX ? 0 : a][0], base + (size_t)(cell - stride[a]) * VB, xi, node) - fi;
      if (has[a][1]) dhi = value(cell + stride[a], stn[FX ? 0 : a][1], base + (size_t)(cell + stride[a]) * VB, xi, node) - fi;
      dp.raise(dlo);
      dp.raise(dhi);
      dn.raise_neg(dlo);
      dn.raise_neg(dhi);
      const T inc = (gc[a].clo * dlo + gc[a].chi * dhi) * ((side & 1) ? gc[a].rhi : gc[a].rlo);
      d2.raise_abs(inc);
      if (a == axn) dout = inc;
    }
    const T face = fi + venkat_phi<T>(dp, dn, d2, eps2) * dout;
    acc += (double)(w * fabs(xa) * face);
  }
  __shared__ double red[256];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) rho_w[wf] = red[0] / Z0[side];
}

template <typename T, typename S>
cudaError_t launch_wall_prepass(const KinArgs<T, S> &a, const int *wall_cell, const int *wall_side, int nwall,
                                const double *Z0, double *rho_w, int nslots, cudaStream_t s) {
  if (nwall == 0) return cudaSuccess;
  auto launch = [&](auto fx) {
    constexpr bool FX = decltype(fx)::value;
    if (a.g.nact == 1) wall_prepass_kernel<T, S, 1, FX><<<nwall, 256, 0, s>>>(a, wall_cell, wall_side, Z0, rho_w, nslots);
    else if (a.g.nact == 2) wall_prepass_kernel<T, S, 2, FX><<<nwall, 256, 0, s>>>(a, wall_cell, wall_side, Z0, rho_w, nslots);
    else wall_prepass_kernel<T, S, 3, FX><<<nwall, 256, 0, s>>>(a, wall_cell, wall_side, Z0, rho_w, nslots);
  };
  if constexpr (std::is_same<T, double>::value) {
    if (a.ftab) launch(std::true_type{});
    else launch(std::false_type{});
  } else {
    launch(std::false_type{});
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Wall constants: for each wall side, over the velocities leaving the wall into the gas,
//   Z0 = sum w |xi_n| M_w  and  Zw[m] = sum w xi_a phi_m M_w (signed, +e_a direction),
// phi = 1, xi(3), |xi|^2/2 and the internal-energy factor d_r T_w / 4 (Rykov).
__global__ void wall_constants_kernel(const double *vel64, int nslots, const double *wall_uT, const int *sides,
                                      double *Z0, double *Zw, double d_r) {
  const int side = sides[blockIdx.x], a = side / 2;
  const double dir = (side & 1) ? 1.0 : -1.0;
  const double *uT = wall_uT + 4 * side;
  double acc[7] = {0, 0, 0, 0, 0, 0, 0};
  const double norm = pow(3.14159265358979323846 * uT[3], -1.5);
  for (int v = threadIdx.x; v < nslots; v += blockDim.x) {
    const double x = vel64[4 * v], y = vel64[4 * v + 1], z = vel64[4 * v + 2], w = vel64[4 * v + 3];
    const double xa = a == 0 ? x : (a == 1 ? y : z);
    if (!(w > 0.0) || !(xa * dir < 0.0)) continue;
    const double cx = x - uT[0], cy = y - uT[1], cz = z - uT[2];
    const double M = norm * exp(-(cx * cx + cy * cy + cz * cz) / uT[3]);
    const double fl = w * xa * M;
    acc[0] += w * fabs(xa) * M;
    acc[1] += fl;
    acc[2] += fl * x;
    acc[3] += fl * y;
    acc[4] += fl * z;
    acc[5] += fl * (0.5 * (x * x + y * y + z * z) + d_r * uT[3] / 4.0);
    acc[6] += fl * d_r * uT[3] / 4.0;
  }
  __shared__ double red[7][256];
  for (int q = 0; q < 7; ++q) red[q][threadIdx.x] = acc[q];
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o)
      for (int q = 0; q < 7; ++q) red[q][threadIdx.x] += red[q][threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    Z0[side] = red[0][0];
    for (int q = 0; q < 6; ++q) Zw[6 * side + q] = red[1 + q][0];
  }
}

cudaError_t launch_wall_constants(const double *vel64, int nslots, const double *wall_uT, const int *sides,
                                  int nsides, double *Z0, double *Zw, double d_r, cudaStream_t s) {
  if (nsides == 0) return cudaSuccess;
  wall_constants_kernel<<<nsides, 256, 0, s>>>(vel64, nslots, wall_uT, sides, Z0, Zw, d_r);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Moments of the stored f (Eq. getmoment) streamed after the kinetic step: one thread owns one
// cell and a chunk of velocity blocks, reads the block's 32 values of its cell as vectors and
// accumulates, about the state velocity u_n,
//   13 raw moments of f (1, c, cc, |c|^2 c)  and  5 moments of w (g^n - f) (1, xi, |xi|^2/2).
// The second set gives, through the discrete identity of the delta-form equation with 1/dt = 0,
//   sum over the cell's faces of the outward kinetic flux = V sum_v w phi (g^n - f^{n+1/2}) / tau,
// the only kinetic-flux information the synthetic solve needs.  Sums over one block (32 terms)
// are plain, and are added into compensated (Kahan) accumulators across blocks.
template <typename T, int N>
struct MomAcc {
  T s[N], c[N];
  __device__ void zero() {
#pragma unroll
    for (int k = 0; k < N; ++k) s[k] = c[k] = (T)0;
  }
  __device__ void add(const T *x) {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const T y = x[k] - c[k];
      const T t = s[k] + y;
      c[k] = (t - s[k]) - y;
      s[k] = t;
    }
  }
};

template <typename T, typename S>
__device__ __forceinline__ void load_block_f(const S *p, T *f);
template <>
__device__ __forceinline__ void load_block_f<float, float>(const float *p, float *f) {
  const float4 *q = reinterpret_cast<const float4 *>(p);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 v = __ldcs(q + i);
    f[4 * i] = v.x;
    f[4 * i + 1] = v.y;
    f[4 * i + 2] = v.z;
    f[4 * i + 3] = v.w;
  }
}
template <>
__device__ __forceinline__ void load_block_f<float, __nv_bfloat16>(const __nv_bfloat16 *p, float *f) {
  const uint4 *q = reinterpret_cast<const uint4 *>(p);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint4 v = __ldcs(q + i);
    const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      // a 32-bit word holds two BF16 values, the lower-addressed one in the low half; a BF16
      // value is the upper 16 bits of the FP32 value it widens to
      f[8 * i + 2 * j] = __uint_as_float(w[j] << 16);
      f[8 * i + 2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
    }
  }
}
template <>
__device__ __forceinline__ void load_block_f<double, double>(const double *p, double *f) {
  const double2 *q = reinterpret_cast<const double2 *>(p);
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const double2 v = __ldcs(q + i);
    f[2 * i] = v.x;
    f[2 * i + 1] = v.y;
  }
}

template <typename T, typename S, int NV>
__global__ void __launch_bounds__(128) moments_kernel(const KinArgs<T, S> A, int blocks_per_chunk, double *mp) {
  constexpr int NP = moment_len(NV);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *svel = reinterpret_cast<T *>(smem_raw);  // [blocks_per_chunk * VB][4]
  const KinGeom &G = A.g;
  const int chunk = blockIdx.y;
  const int b0 = chunk * blocks_per_chunk;
  const int nb = min(blocks_per_chunk, A.nblocks - b0);
  for (int i = threadIdx.x; i < nb * VB * 4; i += blockDim.x) svel[i] = A.vel[(size_t)b0 * VB * 4 + i];
  __syncthreads();
  const int cell = blockIdx.x * blockDim.x + threadIdx.x;
  if (cell >= G.nc) return;
  constexpr int CL = NV == 2 ? NST_RYKOV : 16;
  T st[CL];
  load_state<CL>(A.st + (size_t)cell * NST, st);
  MomAcc<T, NP> acc;
  acc.zero();
  for (int bb = 0; bb < nb; ++bb) {
    T f[VB], f1[NV == 2 ? VB : 1];
    load_block_f<T, S>(A.f + ((size_t)(b0 + bb) * G.nc + cell) * VB, f);
    if constexpr (NV == 2) load_block_f<T, S>(A.f1 + ((size_t)(b0 + bb) * G.nc + cell) * VB, f1);
    T sum[NP];
#pragma unroll
    for (int k = 0; k < NP; ++k) sum[k] = (T)0;
#pragma unroll
    for (int l = 0; l < VB; ++l) {
      const T *v = svel + (bb * VB + l) * 4;
      const T x = v[0], y = v[1], z = v[2], w = v[3];
      const T cx = x - st[0], cy = y - st[1], cz = z - st[2];
      const T c2 = cx * cx + cy * cy + cz * cz;
      T mw, g[NV];  // Maxwellian of W^n (the storage reference of this step) and the reference
      if constexpr (NV == 1) {
        mw = st[4] * dexp(-c2 * st[3]);
      } else {
        reference<T, NV>(st, cx, cy, cz, c2, mw, g);
      }
      const T wf = w * (StoredRelative<S>::value ? f[l] + mw : f[l]);
      sum[0] += wf;
      sum[1] += wf * cx;
      sum[2] += wf * cy;
      sum[3] += wf * cz;
      sum[4] += wf * cx * cx;
      sum[5] += wf * cy * cy;
      sum[6] += wf * cz * cz;
      sum[7] += wf * cx * cy;
      sum[8] += wf * cx * cz;
      sum[9] += wf * cy * cz;
      sum[10] += wf * c2 * cx;
      sum[11] += wf * c2 * cy;
      sum[12] += wf * c2 * cz;
      T d, d1 = (T)0;
      if constexpr (NV == 1) {
        const T shak = (st[12] * cx + st[13] * cy + st[14] * cz) * (c2 * st[3] - (T)2.5);
        // w (g - f): with relative storage g - f = M shak - (f - M) needs no difference of O(1)
        // values (the sum is multiplied by 1/tau, which at small Kn would amplify that round-off)
        d = StoredRelative<S>::value ? w * (mw * shak - f[l]) : w * (mw * ((T)1 + shak)) - wf;
      } else {
        const T wf1 = w * (StoredRelative<S>::value ? f1[l] + st[29] * mw : f1[l]);
        d = w * g[0] - wf;
        d1 = w * g[NV - 1] - wf1;
        sum[NMOM + NFF + 1] += wf1;
        sum[NMOM + NFF + 2] += wf1 * cx;
        sum[NMOM + NFF + 3] += wf1 * cy;
        sum[NMOM + NFF + 4] += wf1 * cz;
        sum[NMOM + NFF] += d1;
      }
      sum[13] += d;
      sum[14] += d * x;
      sum[15] += d * y;
      sum[16] += d * z;
      sum[17] += d * (T)0.5 * (x * x + y * y + z * z) + d1;
    }
    acc.add(sum);
  }
  double *out = mp + ((size_t)chunk * G.nc + cell) * NP;
#pragma unroll
  for (int k = 0; k < NP; ++k) out[k] = (double)acc.s[k] - (double)acc.c[k];
}

template <typename T, typename S>
cudaError_t launch_moments(const KinArgs<T, S> &a, int blocks_per_chunk, int nchunks, double *mp, cudaStream_t s) {
  const size_t smem = (size_t)blocks_per_chunk * VB * 4 * sizeof(T);
  auto k = a.nvdf == 2 ? moments_kernel<T, S, 2> : moments_kernel<T, S, 1>;
  // (the same limit for every solver: see kinetic_shape)
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, MOM_MAX_BLOCKS * VB * 4 * (int)sizeof(T));
  if (e != cudaSuccess) return e;
  dim3 grid((a.g.nc + 127) / 128, nchunks);
  k<<<grid, 128, smem, s>>>(a, blocks_per_chunk, mp);
  return cudaGetLastError();
}

struct __align__(16) double4_16 {
  double x, y, z, w;
};

// FP64 storage on a tensor-product grid, Shakhov: the 13 moments of the stored f^{n+1/2} about the origin,
// w (1, xi(3), xi_a xi_b (6), |xi|^2 xi(3)), no exponential.  The collision sums sum_v w phi (g^n - f) are
// assembled per cell by the reduction from the closed form of sum_v w phi g^n (ref_sums_kernel) and
// these moments.  Row layout as in moments_kernel.  Both cancel where |u| is many thermal speeds (the
// heat flux loses a factor of |u|^3), so the two VDFs of Rykov, the gas of the hypersonic cases, keep
// moments_kernel: about the state velocity, with g - f formed point by point (cavity 48^2 with 20^3
// velocities, moments and reductions 3.8 ms; this form took 0.8).

// Untiled grids: from the per-slot table of the 13 factors (16 doubles per slot, the last three 0),
// one FMA per moment and point.  Per-block plain sums, compensated (Kahan) across the chunk's blocks.
__global__ void __launch_bounds__(128) moments_origin_kernel(const KinArgs<double, double> A, const double *mtab,
                                                             int blocks_per_chunk, double *mp) {
  constexpr int NP = moment_len(1);
  const int chunk = blockIdx.y;
  const int b0 = chunk * blocks_per_chunk;
  const int nb = min(blocks_per_chunk, A.nblocks - b0);
  const int cell = blockIdx.x * blockDim.x + threadIdx.x;
  if (cell >= A.g.nc) return;
  MomAcc<double, NMOM> acc;
  acc.zero();
  for (int bb = 0; bb < nb; ++bb) {
    double f[VB];
    load_block_f<double, double>(A.f + ((size_t)(b0 + bb) * A.g.nc + cell) * VB, f);
    const double2 *tb = reinterpret_cast<const double2 *>(mtab + (size_t)(b0 + bb) * VB * 16);
    double sum[NMOM];
#pragma unroll
    for (int k = 0; k < NMOM; ++k) sum[k] = 0.0;
#pragma unroll
    for (int l = 0; l < VB; ++l) {
      double t[14];
#pragma unroll
      for (int q = 0; q < 7; ++q) {
        const double2 v = __ldg(tb + l * 8 + q);
        t[2 * q] = v.x;
        t[2 * q + 1] = v.y;
      }
#pragma unroll
      for (int k = 0; k < NMOM; ++k) sum[k] = fma(f[l], t[k], sum[k]);
    }
    acc.add(sum);
  }
  double *out = mp + ((size_t)chunk * A.g.nc + cell) * NP;
#pragma unroll
  for (int k = 0; k < NP; ++k) out[k] = 0.0;
#pragma unroll
  for (int k = 0; k < NMOM; ++k) out[k] = acc.s[k] - acc.c[k];
}

// Tiled grids: a block of 32 velocities is a TX x TY x TZ tile, so its sums factorise: over x with
// the powers 0..3 of the node (btab [block][node of x, y, z][4]: w, w xi, w xi^2, w xi^3 per axis),
// then over y, then over z: 246 FP64 instructions per tile instead of 416 (4 per point for x, the
// rest on 8 and 2 values).  Plain sums over four tiles (at most 14 additions deep), compensated
// across them.  The FP64 pipe bounds it: 128^2 cells with 32^3 velocities 13.6 -> 7.8 ms with the
// reductions.
template <int TX, int TY, int TZ>
__global__ void __launch_bounds__(128) moments_tile_kernel(const KinArgs<double, double> A, const double *btab,
                                                           int blocks_per_chunk, double *mp) {
  constexpr int NP = moment_len(1), NN = TX + TY + TZ;
  const int chunk = blockIdx.y;
  const int b0 = chunk * blocks_per_chunk;
  const int nb = min(blocks_per_chunk, A.nblocks - b0);
  const int cell = blockIdx.x * blockDim.x + threadIdx.x;
  if (cell >= A.g.nc) return;
  MomAcc<double, NMOM> acc;
  acc.zero();
  double S[NMOM];
#pragma unroll
  for (int k = 0; k < NMOM; ++k) S[k] = 0.0;
  for (int bb = 0; bb < nb; ++bb) {
    const size_t at = ((size_t)(b0 + bb) * A.g.nc + cell) * VB;
    const double4_16 *tab = reinterpret_cast<const double4_16 *>(btab + (size_t)(b0 + bb) * NN * 4);
    double4_16 tx[TX];
#pragma unroll
    for (int i = 0; i < TX; ++i) tx[i] = tab[i];
#pragma unroll
    for (int iz = 0; iz < TZ; ++iz) {
      // sums over x and y of f times x^p y^q, p + q <= 3
      double B[4][4];
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) B[p][q] = 0.0;
#pragma unroll
      for (int iy = 0; iy < TY; ++iy) {
        const int l = TX * (iy + TY * iz);
        const double4_16 ty = tab[TX + iy];
        const double py[4] = {ty.x, ty.y, ty.z, ty.w};
        double a[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int ix = 0; ix < TX; ix += 2) {
          const double2 v = __ldcs(reinterpret_cast<const double2 *>(A.f + at + l + ix));
          a[0] = fma(v.y, tx[ix + 1].x, fma(v.x, tx[ix].x, a[0]));
          a[1] = fma(v.y, tx[ix + 1].y, fma(v.x, tx[ix].y, a[1]));
          a[2] = fma(v.y, tx[ix + 1].z, fma(v.x, tx[ix].z, a[2]));
          a[3] = fma(v.y, tx[ix + 1].w, fma(v.x, tx[ix].w, a[3]));
        }
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int q = 0; p + q < 4; ++q) B[p][q] = fma(a[p], py[q], B[p][q]);
      }
      const double4_16 z = tab[TX + TY + iz];
      S[0] = fma(B[0][0], z.x, S[0]);
      S[1] = fma(B[1][0], z.x, S[1]);
      S[2] = fma(B[0][1], z.x, S[2]);
      S[3] = fma(B[0][0], z.y, S[3]);
      S[4] = fma(B[2][0], z.x, S[4]);
      S[5] = fma(B[0][2], z.x, S[5]);
      S[6] = fma(B[0][0], z.z, S[6]);
      S[7] = fma(B[1][1], z.x, S[7]);
      S[8] = fma(B[1][0], z.y, S[8]);
      S[9] = fma(B[0][1], z.y, S[9]);
      S[10] = fma(B[1][0], z.z, fma(B[3][0] + B[1][2], z.x, S[10]));
      S[11] = fma(B[0][1], z.z, fma(B[2][1] + B[0][3], z.x, S[11]));
      S[12] = fma(B[0][0], z.w, fma(B[2][0] + B[0][2], z.y, S[12]));
    }
    if ((bb & 3) == 3 || bb == nb - 1) {
      acc.add(S);
#pragma unroll
      for (int k = 0; k < NMOM; ++k) S[k] = 0.0;
    }
  }
  double *out = mp + ((size_t)chunk * A.g.nc + cell) * NP;
#pragma unroll
  for (int k = 0; k < NP; ++k) out[k] = 0.0;
#pragma unroll
  for (int k = 0; k < NMOM; ++k) out[k] = acc.s[k] - acc.c[k];
}

// Closed form of sum_v w phi(xi) g^n(xi), phi = 1, xi(3), |xi|^2/2, on a tensor-product velocity grid:
// with c = xi - u the Shakhov distribution C e^{-|c|^2/T} [1 + a.c (|c|^2/T - 5/2)] is a polynomial in c
// times a product of one-dimensional Gaussians, so the sum over the grid factorises into the
// one-dimensional sums m_a[k] = sum_i w_a(i) e^{-c_a(i)^2/T} c_a(i)^k (k <= 5; C in the x ones).  Per
// cell 3 lanes take one axis each, then one writes the cell's row of the extra moment chunk (moments
// 0, collision sums after them); emit = 0 (the velocity shards other than the first) writes zeros, so
// the sum over shards counts it once.
__global__ void __launch_bounds__(96) ref_sums_kernel(int nc, const double *st64, const double *vaxis, int nx, int ny,
                                                           int nz, int emit, double *row) {
  constexpr int NP = moment_len(1);
  __shared__ double m[3][6][33];
  const int slot = threadIdx.x & 31, a = threadIdx.x >> 5;
  const int cell = blockIdx.x * 32 + slot;
  const double *st = st64 + (size_t)cell * NST;
  if (cell < nc && emit) {
    const int n = a == 0 ? nx : (a == 1 ? ny : nz);
    const double *x = vaxis + (a == 0 ? 0 : (a == 1 ? nx : nx + ny)), *w = x + nx + ny + nz;
    const double u = st[a], invT = st[3];
    double s[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int i = 0; i < n; ++i) {
      const double c = x[i] - u;
      double p = w[i] * exp(-c * c * invT);
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        s[k] += p;
        p *= c;
      }
    }
    const double C = a == 0 ? st[4] : 1.0;
#pragma unroll
    for (int k = 0; k < 6; ++k) m[a][k][slot] = C * s[k];
  }
  __syncthreads();
  if (a != 0 || cell >= nc) return;
  double *o = row + (size_t)cell * NP;
#pragma unroll
  for (int k = 0; k < NP; ++k) o[k] = 0.0;
  if (!emit) return;
  const double u[3] = {st[0], st[1], st[2]};
  auto mono = [&](int px, int py, int pz) { return m[0][px][slot] * m[1][py][slot] * m[2][pz][slot]; };
  const double invT = st[3], *aq = st + 12;
  // sum_v w g c^e for the exponent triple e
  auto G = [&](int px, int py, int pz) {
    double t1 = 0.0;
    for (int b = 0; b < 3; ++b) {
      const int e[3] = {px + (b == 0), py + (b == 1), pz + (b == 2)};
      const double s3 = mono(e[0] + 2, e[1], e[2]) + mono(e[0], e[1] + 2, e[2]) + mono(e[0], e[1], e[2] + 2);
      t1 += aq[b] * (invT * s3 - 2.5 * mono(e[0], e[1], e[2]));
    }
    return mono(px, py, pz) + t1;
  };
  const double g1 = G(0, 0, 0);
  const double gc[3] = {G(1, 0, 0), G(0, 1, 0), G(0, 0, 1)};
  const double gc2 = G(2, 0, 0) + G(0, 2, 0) + G(0, 0, 2);
  o[NMOM] = g1;
  for (int b = 0; b < 3; ++b) o[NMOM + 1 + b] = gc[b] + u[b] * g1;
  o[NMOM + 4] = 0.5 * gc2 + (u[0] * gc[0] + u[1] * gc[1] + u[2] * gc[2]) +
                0.5 * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]) * g1;
}

cudaError_t launch_moments_origin(const KinArgs<double, double> &a, const double *mtab, int blocks_per_chunk,
                                  int nchunks, const double *st64, const double *vaxis, const int *nv_axis, int emit,
                                  double *mp, cudaStream_t s) {
  dim3 grid((a.g.nc + 127) / 128, nchunks);
  void (*k)(const KinArgs<double, double>, const double *, int, double *) =
      a.g.tile[0] == 0   ? moments_origin_kernel
      : a.g.tile[0] == 2 ? moments_tile_kernel<2, 4, 4>
      : a.g.tile[1] == 2 ? moments_tile_kernel<4, 2, 4>
                         : moments_tile_kernel<4, 4, 2>;
  k<<<grid, 128, 0, s>>>(a, mtab, blocks_per_chunk, mp);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  ref_sums_kernel<<<(a.g.nc + 31) / 32, 96, 0, s>>>(a.g.nc, st64, vaxis, nv_axis[0], nv_axis[1], nv_axis[2], emit,
                                                    mp + (size_t)nchunks * a.g.nc * moment_len(1));
  return cudaGetLastError();
}

// f_raw = Maxwellian(W0) of each cell at each slot velocity, in the storage precision (the
// per-cell factor rho (pi T)^(-3/2) and 1/T in FP64, the exponential in T).  Relative (BF16,
// FP32) storage writes zero deviations from M(W0), which the initial state names as the
// reference.
__device__ __forceinline__ float accurate_exp(float x) { return expf(x); }
__device__ __forceinline__ double accurate_exp(double x) { return exp(x); }

// One warp per cell: the per-cell factors once (FP64 is scarce on this GPU), then every
// velocity block of the cell, one 128-byte line per block.
template <typename T, typename S>
__global__ void init_maxwellian_kernel(const KinArgs<T, S> A, const double *W0) {
  const KinGeom &G = A.g;
  const int lane = threadIdx.x & 31;
  const int cell = (int)(((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (cell >= G.nc) return;
  const double *w0 = W0 + 6 * (size_t)cell;
  const T C = (T)(w0[0] * pow(3.14159265358979323846 * w0[4], -1.5)), invT = (T)(1.0 / w0[4]);
  const T ux = (T)w0[1], uy = (T)w0[2], uz = (T)w0[3];
  const T c1 = (T)(A.d_r * w0[5] / 4.0);  // f1 = (d_r Tr / 4) f0 (Rykov)
  for (int b = 0; b < A.nblocks; ++b) {
    const T *vp = A.vel + ((size_t)b * VB + lane) * 4;
    const T cx = vp[0] - ux, cy = vp[1] - uy, cz = vp[2] - uz;
    // relative storage: f is exactly the reference Maxwellian M(W0), stored as a zero deviation
    const T f = StoredRelative<S>::value ? (T)0 : C * accurate_exp(-(cx * cx + cy * cy + cz * cz) * invT);
    Fio<T, S>::st(A.f + ((size_t)b * G.nc + cell) * VB + lane, f);
    if (A.nvdf == 2) Fio<T, S>::st(A.f1 + ((size_t)b * G.nc + cell) * VB + lane, c1 * f);
  }
}

template <typename T, typename S>
cudaError_t launch_init_maxwellian(const KinArgs<T, S> &a, const double *W0, int nblocks, cudaStream_t s) {
  (void)nblocks;
  const int threads = 256;
  const size_t grid = ((size_t)a.g.nc * 32 + threads - 1) / threads;
  init_maxwellian_kernel<T, S><<<(unsigned)grid, threads, 0, s>>>(a, W0);
  return cudaGetLastError();
}

// Canonical [cell][v] FP64 <-> internal [block][cell][lane].  Export applies the pending
// correction (the returned f is the VDF the next kinetic step starts from).
template <typename T, typename S>
__global__ void export_f_kernel(const KinArgs<T, S> A, int q, const int *slot_canon, int nslots, int nv, double *out) {
  const size_t n = (size_t)A.g.nc * nslots;
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < n; idx += (size_t)gridDim.x * blockDim.x) {
    const int slot = (int)(idx % nslots);
    const int cell = (int)(idx / nslots);
    const T *vp = A.vel + (size_t)slot * 4;
    if (!(vp[3] > (T)0)) continue;
    T st[NST_RYKOV];
    load_state<NST_RYKOV>(A.st + (size_t)cell * NST, st);
    const int blk = slot / VB, ln = slot % VB;
    const size_t at = ((size_t)blk * A.g.nc + cell) * VB + ln;
    T stored[2] = {Fio<T, S>::ld(A.f + at), (T)0}, f[2];
    if (A.nvdf == 2) {
      stored[1] = Fio<T, S>::ld(A.f1 + at);
      corrected_all<T, S, 2>(stored, st, vp[0], vp[1], vp[2], f);
    } else {
      corrected_all<T, S, 1>(stored, st, vp[0], vp[1], vp[2], f);
    }
    out[(size_t)cell * nv + slot_canon[slot]] = (double)f[q];
  }
}

template <typename T, typename S>
__global__ void import_f_kernel(const KinArgs<T, S> A, int q, const int *slot_canon, int nslots, int nv, const double *in) {
  const size_t n = (size_t)A.g.nc * nslots;
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < n; idx += (size_t)gridDim.x * blockDim.x) {
    const int slot = (int)(idx % nslots);
    const int cell = (int)(idx / nslots);
    const int blk = slot / VB, ln = slot % VB;
    Fio<T, S>::st((q ? A.f1 : A.f) + ((size_t)blk * A.g.nc + cell) * VB + ln, (T)in[(size_t)cell * nv + slot_canon[slot]]);
  }
}

template <typename T, typename S>
cudaError_t launch_export_f(const KinArgs<T, S> &a, int q, const int *slot_canon, int nslots, int nv, double *out,
                            cudaStream_t s) {
  export_f_kernel<T, S><<<1024, 256, 0, s>>>(a, q, slot_canon, nslots, nv, out);
  return cudaGetLastError();
}

template <typename T, typename S>
cudaError_t launch_import_f(const KinArgs<T, S> &a, int q, const int *slot_canon, int nslots, int nv, const double *in,
                            cudaStream_t s) {
  import_f_kernel<T, S><<<1024, 256, 0, s>>>(a, q, slot_canon, nslots, nv, in);
  return cudaGetLastError();
}

#define GSIS_INST(T, S)                                                                                         \
  template cudaError_t launch_kinetic<T, S>(const KinArgs<T, S> &, int, int, size_t, cudaStream_t);             \
  template cudaError_t kinetic_shape<T, S>(const KinGeom &, int, bool, bool, int, size_t, int *, int *);                                       \
  template cudaError_t launch_wall_prepass<T, S>(const KinArgs<T, S> &, const int *, const int *, int,           \
                                                 const double *, double *, int, cudaStream_t);                   \
  template cudaError_t launch_moments<T, S>(const KinArgs<T, S> &, int, int, double *, cudaStream_t);           \
  template cudaError_t launch_init_maxwellian<T, S>(const KinArgs<T, S> &, const double *, int, cudaStream_t);   \
  template cudaError_t launch_export_f<T, S>(const KinArgs<T, S> &, int, const int *, int, int, double *,       \
                                             cudaStream_t);                                                      \
  template cudaError_t launch_import_f<T, S>(const KinArgs<T, S> &, int, const int *, int, int, const double *, \
                                             cudaStream_t);
GSIS_INST(float, float)
GSIS_INST(double, double)
GSIS_INST(float, __nv_bfloat16)
template size_t kinetic_smem_bytes<float, float>(const KinGeom &, int);
template size_t kinetic_smem_bytes<double, double>(const KinGeom &, int);
template size_t kinetic_smem_bytes<float, __nv_bfloat16>(const KinGeom &, int);
template size_t kinetic_gscratch_stride<float, float>(const KinGeom &, int);
template size_t kinetic_gscratch_stride<double, double>(const KinGeom &, int);
template size_t kinetic_gscratch_stride<float, __nv_bfloat16>(const KinGeom &, int);

}  // namespace gsis
