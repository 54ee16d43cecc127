// Incident-wave boundary data and field evaluation from point strengths.
//
// Incident data (Sec. 2 eqs. ui, neu; Sec. 3.4 eq. trans) is sampled on the
// M x P ring nodes (rho_m, phi_l = 2 pi l / P, z_m) that the RHS transform
// (eq. fhatquad with q = P) consumes.
//
// Field evaluation (Sec. 4.1): each ring source of mode n is replaced by P
// point sources with strengths sigma_jl (the inverse transform of c_nj over
// n), so u(x) = sum_{j,l} G_k(x, y_jl) sigma_jl. With a lattice the sum runs
// over the eight phased nearest images, the action A_else of Sec. 4.1 done by
// direct summation instead of an FMM.
#include <cooperative_groups.h>

#include "axi_internal.h"
#include "trig.cuh"

namespace cg = cooperative_groups;

namespace axi {
namespace {

constexpr int kThreads = 256;
constexpr double kInv4Pi = 0.07957747154594766788;

__global__ void incident_kernel(const ObsDev *__restrict__ od, int W, const double *__restrict__ dirs,
                                double2 *__restrict__ f) {
  const ObsDev &o = *od;
  const int P = o.P, rows = o.rows;
  const size_t total = (size_t)W * rows * P;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    const int l = (int)(e % P);
    const int row = (int)((e / P) % rows);
    const int w = (int)(e / ((size_t)P * rows));
    const int m = row % o.M;
    const double rho = o.coll[4 * m], z = o.coll[4 * m + 1];
    const double nr = o.coll[4 * m + 2], nz = o.coll[4 * m + 3];
    const double2 t = o.tw_P[l];       // (cos phi_l, -sin phi_l)
    const double c = t.x, s = -t.y;
    const double dx = dirs[3 * w], dy = dirs[3 * w + 1], dz = dirs[3 * w + 2];
    const double dxv = dx * rho * c + dy * rho * s + dz * z;     // d . x
    const double dnv = dx * nr * c + dy * nr * s + dz * nz;      // d . n
    double sn, cs;
    sincos(o.k * dxv, &sn, &cs);
    double2 v;
    const bool value_row = (o.bc == AXI_BC_TRANSMISSION) && row < o.M;
    if (value_row) {
      v = make_double2(-cs, -sn);                              // -u_i
    } else {
      const double a = o.k * dnv;                              // -du/dn = -i k (d.n) u_i
      v = make_double2(a * sn, -a * cs);
    }
    f[e] = v;
  }
}

__device__ const long long g_field_ring_q62[trig::kRingTab][2] = {
#include "ring_table_q62.inc"
};

// Kernel value times 4 pi: e^{ikR}/R, its normal derivative, or e^{-ik x.y}.
// The FP64 pipe bounds the evaluation (1/64 rate), so the square root comes
// from rsqrt with one correction (a division and a square root cost twice
// that), and the phase, sin and cos run in fixed point (trig::sincos_phase):
// 16 FP64 operations for the potential.
template <int KIND>
__device__ __forceinline__ double2 field_kernel(const trig::RingPhase &ph, double tx, double ty, double tz, double nx,
                                                double ny, double nz, double yx, double yy, double yz) {
  const longlong2 *tab = reinterpret_cast<const longlong2 *>(g_field_ring_q62);   // through L1
  const trig::PhaseOffset none{0, 0};
  double sn, cs;
  if (KIND == AXI_EVAL_FAR_FIELD) {
    const double a = fma(tx, yx, fma(ty, yy, tz * yz));
    trig::sincos_phase(fabs(a), ph, none, tab, &sn, &cs);
    // -sin(k a) = -sign(a) sin(k |a|), on the bits
    return make_double2(cs, __longlong_as_double(__double_as_longlong(sn) ^
                                                 (~__double_as_longlong(a) & (long long)(1ull << 63))));
  }
  const double dx = tx - yx, dy = ty - yy, dz = tz - yz;
  const double R2 = fma(dx, dx, fma(dy, dy, dz * dz));
  const double inv = rsqrt(R2);
  double R = R2 * inv;
  R = fma(0.5 * inv, fma(-R, R, R2), R);                   // to half a unit in the last place
  trig::sincos_phase(R, ph, none, tab, &sn, &cs);
  if (KIND == AXI_EVAL_POTENTIAL) return make_double2(cs * inv, sn * inv);
  const double f = fma(nx, dx, fma(ny, dy, nz * dz)) * (inv * inv) * inv, kR = ph.k * R;
  return make_double2(f * fma(-kR, sn, -cs), f * fma(kR, cs, -sn));   // (ikR - 1) e^{ikR}
}

// A cluster of CTAs per target and group of NW waves (grid.x = targets x
// cluster size): the CTAs' threads stride over the sources s = (j, l) of the
// exterior field (first N columns) and, with a lattice, over the eight images.
// A kernel value is formed once per (target, source, image) and used for the
// group's waves, NW chosen to fit them (a fixed group of 8 spent 32 FP64
// operations a value on phases and sums of waves that were not there: the
// potential at 4096 targets of 21600 sources, 4 waves, took 12.9 ms and now takes
// 5.2). The partial sums of a cluster are added by its first CTA in rank order.
constexpr int kWG = 16;
template <int KIND, int NW, bool LAT>
__global__ void __launch_bounds__(kThreads)
eval_kernel(const ObsDev *__restrict__ od, int W, const double2 *__restrict__ sigma, int T,
            const double *__restrict__ targets, const double *__restrict__ normals, double ex, double ey,
            const double *__restrict__ dirs, double2 *__restrict__ out) {
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const ObsDev &o = *od;
  const int t = blockIdx.x / C;
  const int w0 = blockIdx.y * NW;
  const int nw = min(NW, W - w0);
  const int P = o.P, cols = o.cols;
  const double tx = targets[3 * t], ty = targets[3 * t + 1], tz = targets[3 * t + 2];
  const trig::RingPhase ph = o.ph;
  double nx = 0, ny = 0, nz = 0;
  if (KIND == AXI_EVAL_NORMAL_DERIV) { nx = normals[3 * t]; ny = normals[3 * t + 1]; nz = normals[3 * t + 2]; }
  __shared__ double2 phase[LAT ? NW : 1][9];
  if (LAT) {
    for (int e = threadIdx.x; e < NW * 9; e += kThreads) {
      const int w = e / 9, im = e % 9;
      double sn = 0.0, cs = 0.0;
      if (w < nw)
        sincos(ph.k * (dirs[3 * (w0 + w)] * (im / 3 - 1) * ex + dirs[3 * (w0 + w) + 1] * (im % 3 - 1) * ey), &sn, &cs);
      phase[w][im] = make_double2(cs, sn);
    }
    __syncthreads();
  }
  double2 acc[NW];
#pragma unroll
  for (int w = 0; w < NW; ++w) acc[w] = make_double2(0.0, 0.0);
  const int S = o.N * P, step = C * kThreads, dj = step / P, dl = step % P;
  int s = rank * kThreads + threadIdx.x, j = s / P, l = s % P;
  for (; s < S; s += step) {
    const double2 tw = o.tw_P[l];
    const double rs = o.src[2 * j], yz = o.src[2 * j + 1];
    const double yx = rs * tw.x, yy = -rs * tw.y;
    const double2 *sg = sigma + ((size_t)w0 * cols + j) * P + l;
    double2 val[LAT ? NW : 1];
    if (LAT) {
#pragma unroll
      for (int w = 0; w < NW; ++w) val[w] = make_double2(0.0, 0.0);
      for (int im = 0; im < 9; ++im) {
        if (im == 4) continue;                             // central copy excluded (A_else)
        const double2 kv = field_kernel<KIND>(ph, tx, ty, tz, nx, ny, nz, yx + (im / 3 - 1) * ex,
                                              yy + (im % 3 - 1) * ey, yz);
#pragma unroll
        for (int w = 0; w < NW; ++w) {
          const double2 ph = phase[w][im];
          val[w].x = fma(ph.x, kv.x, fma(-ph.y, kv.y, val[w].x));
          val[w].y = fma(ph.x, kv.y, fma(ph.y, kv.x, val[w].y));
        }
      }
    } else {
      val[0] = field_kernel<KIND>(ph, tx, ty, tz, nx, ny, nz, yx, yy, yz);
    }
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      if (w < nw) {
        const double2 g = sg[(size_t)w * cols * P], v = val[LAT ? w : 0];
        acc[w].x = fma(v.x, g.x, fma(-v.y, g.y, acc[w].x));
        acc[w].y = fma(v.x, g.y, fma(v.y, g.x, acc[w].y));
      }
    }
    j += dj;
    l += dl;
    if (l >= P) { l -= P; ++j; }
  }
  __shared__ double red[kThreads / 32][2 * NW];
  __shared__ double part[2 * NW];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    // both components in five additions a lane
    const bool up = lane & 16;
    double v = (up ? acc[w].y : acc[w].x) + __shfl_xor_sync(0xffffffffu, up ? acc[w].x : acc[w].y, 16);
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((lane & 15) == 0) red[warp][2 * w + (lane >> 4)] = v;
  }
  __syncthreads();
  if (threadIdx.x < 2 * NW) {
    double v = 0.0;
    for (int i = 0; i < kThreads / 32; ++i) v += red[i][threadIdx.x];
    part[threadIdx.x] = v;
  }
  cluster.sync();
  if (rank == 0 && threadIdx.x < 2 * nw) {
    double v = 0.0;
    for (int r = 0; r < C; ++r) v += cluster.map_shared_rank(part, r)[threadIdx.x];
    reinterpret_cast<double *>(out + (size_t)(w0 + threadIdx.x / 2) * T + t)[threadIdx.x & 1] =
        v * kInv4Pi;
  }
  cluster.sync();                                          // part stays until the first CTA has read it
}

}  // namespace

cudaError_t launch_incident(const ObsDev *d_o, const ObsDev &h, int W, const double *dirs,
                            double2 *f, cudaStream_t st) {
  const size_t total = (size_t)W * h.rows * h.P;
  int blocks = (int)((total + kThreads - 1) / kThreads);
  if (blocks > 152 * 16) blocks = 152 * 16;
  if (blocks < 1) blocks = 1;
  incident_kernel<<<blocks, kThreads, 0, st>>>(d_o, W, dirs, f);
  return cudaGetLastError();
}

namespace {

template <int KIND, int NW, bool LAT>
cudaError_t eval_launch(const ObsDev *d_o, const ObsDev &h, int W, const double2 *sigma, int T,
                        const double *targets, const double *normals, const axi_lattice *lat,
                        const double *dirs, double2 *out, cudaStream_t st) {
  const int groups = (W + NW - 1) / NW;
  // CTAs per target: enough for two a multiprocessor, each with two sources a
  // thread or more
  int C = 1;
  while (C < 8 && (long long)T * groups * C < 2 * sm_count() && (long long)h.N * h.P >= 4LL * C * kThreads) C *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)T * C, (unsigned)groups);
  cfg.blockDim = dim3(kThreads);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, eval_kernel<KIND, NW, LAT>, d_o, W, sigma, T, targets, normals,
                            lat ? lat->ex : 0.0, lat ? lat->ey : 0.0, dirs, out);
}

template <int KIND, bool LAT>
cudaError_t eval_waves(const ObsDev *d_o, const ObsDev &h, int W, const double2 *sigma, int T,
                       const double *targets, const double *normals, const axi_lattice *lat,
                       const double *dirs, double2 *out, cudaStream_t st) {
  if (W <= 1) return eval_launch<KIND, 1, LAT>(d_o, h, W, sigma, T, targets, normals, lat, dirs, out, st);
  if (W <= 2) return eval_launch<KIND, 2, LAT>(d_o, h, W, sigma, T, targets, normals, lat, dirs, out, st);
  if (W <= 4) return eval_launch<KIND, 4, LAT>(d_o, h, W, sigma, T, targets, normals, lat, dirs, out, st);
  if (W <= 8 || LAT) return eval_launch<KIND, 8, LAT>(d_o, h, W, sigma, T, targets, normals, lat, dirs, out, st);
  return eval_launch<KIND, LAT ? 8 : kWG, LAT>(d_o, h, W, sigma, T, targets, normals, lat, dirs, out, st);
}

}  // namespace

cudaError_t launch_eval(const ObsDev *d_o, const ObsDev &h, int W, const double2 *sigma, int T,
                        const double *targets, const double *normals, int kind,
                        const axi_lattice *lat, const double *dirs, double2 *out,
                        cudaStream_t st) {
#define AXI_EVAL(K)                                                                                   \
  return lat ? eval_waves<K, true>(d_o, h, W, sigma, T, targets, normals, lat, dirs, out, st)         \
             : eval_waves<K, false>(d_o, h, W, sigma, T, targets, normals, lat, dirs, out, st)
  if (kind == AXI_EVAL_FAR_FIELD) AXI_EVAL(AXI_EVAL_FAR_FIELD);
  if (kind == AXI_EVAL_NORMAL_DERIV) AXI_EVAL(AXI_EVAL_NORMAL_DERIV);
  AXI_EVAL(AXI_EVAL_POTENTIAL);
#undef AXI_EVAL
}

}  // namespace axi
