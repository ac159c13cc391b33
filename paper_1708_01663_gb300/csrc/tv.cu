// prox of gamma R, R = tau TV_iso + chi_C (Eq. 8), by the fast gradient
// projection (FGP) method of Beck and Teboulle (IEEE TIP 2009), which the
// paper cites for this prox (Sec. III-A) without restating it.  On the dual
// p = (p_x, p_y), with lam = gamma tau, D the forward difference (zero at the
// last index) and P_C the box clamp:
//     x(r)    = P_C(z - lam D^T r)
//     p_k     = Pi_unit-disk(r_k + D x(r_k) / (8 lam))
//     t_{k+1} = (1 + sqrt(1 + 4 t_k^2)) / 2
//     r_{k+1} = p_k + ((t_k - 1) / t_{k+1}) (p_k - p_{k-1})
// from r_1 = p_0 = 0, t_1 = 1; output x(p_K).  2D: several iterations per
// kernel on image tiles with a halo (tv_block_kernel); 3D: one kernel per
// iteration (r ping-pongs between two buffers; p is updated in place per
// pixel), the right neighbour's x by warp shuffle.  Complex f
// takes the separable prox: Re and Im planes, each with its own box.
// The last kernel also applies the relaxed-FISTA momentum of Eq. 11,
// s_{k+1} = f_k + beta (f_k - f_{k-1}).
// 3D volumes take the same iteration with p = (p_x, p_y, p_z), the unit-ball
// projection in R^3 and the dual step 1 / (12 lam) (||D||^2 <= 4 d).
//
// Anisotropic TV (tv_kind 1): R = tau sum_d sum_n |[D_d x]_n| + chi_C, the
// alternative Sec. III-A points to (Kamilov, IEEE TIP 2017).  Along each axis
// the differences split into pairs (i, i+1) with i even and with i odd; each
// parity is a sum over disjoint pairs whose prox keeps the pair's mean and
// soft-thresholds its difference by 2c.  With the box, m = 2d + 1 pieces f_j,
// and prox_{sum f_j}(z) comes from the parallel Dykstra-like proximal
// iteration (Combettes and Pesquet 2011): z_j = z; repeat p_j = prox_{m f_j}(z_j),
// x = mean_j p_j, z_j += x - p_j.  Every step is pointwise (a pixel needs its
// pair partner along each axis), so one kernel per iteration, ping-ponging the
// 2d + 1 auxiliary images between two buffers.
#include <math.h>

#include "common.cuh"

namespace cisor {

// z as planes and, for the 3D iterations, r = p = 0 (r null: none follow).  Dual planes: component k of plane c at
// (3 c + k) * N.
__global__ void tv_split_kernel(const float2* __restrict__ z, float* __restrict__ zp, float* __restrict__ r,
                                float* __restrict__ p, long long N, int ncomp) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const float2 v = z[i];
  zp[i] = v.x;
  if (ncomp == 2) zp[N + i] = v.y;
  if (!r) return;
  for (int k = 0; k < 3 * ncomp; ++k) {
    r[k * N + i] = 0.f;
    p[k * N + i] = 0.f;
  }
}

// Several FGP iterations of a 2D image per launch.  A CTA loads a TVR x TVR region of z, r and p, one pixel a
// thread, runs k iterations on it in shared memory and registers and stores the part that its halo of k pixels
// (k + 1 with the output step) kept exact: one iteration reads r one pixel to the left and above and x one pixel to
// the right and below.  The pixel arithmetic does not depend on the tiling, so neighbouring CTAs agree on what they
// both compute.  Pixels outside the image hold r = 0, which is what the differences' boundary terms need (r is also
// 0 at the last index of its own direction, where the difference is zero).
// One launch per iteration spent 5 us on launch and memory latency for 1 us of arithmetic: 20 iterations of a
// complex 256 x 256 image took 118 us as a call and now take 45 us (real 64 x 64: 99 -> 30 us).  What is left is
// the latency of the iterations themselves (two barriers, a square root and two divisions, 0.4 us each).  More
// iterations a launch (7, 10) recompute more halo than the launches cost at 256 x 256 (61 and 115 us); wider
// regions with several pixels a thread (48 x 48, 64 x 64) leave too few threads to hide the divisions (64 to 84 us).
constexpr int TVR = 32;      // region side, halo included; TVR^2 threads
constexpr int TV_KMAX = 6;   // most iterations of a launch

struct TvBlock {
  const float2* z;       // the prox argument
  const float *rin, *pin;
  float *rout, *pout;    // dual planes (2 c + direction) N
  int n, k, first, last; // first: r = p = 0; last: the output x(p) instead of r and p
  float lam, step, lo[2], hi[2], beta[TV_KMAX];
  int ncomp;             // 1: Im x = 0
  float2* x;
  const float2* fprev;
  float beta_mom;
  float2* s_out;
};

__global__ void __launch_bounds__(TVR* TVR) tv_block_kernel(const TvBlock a) {
  // a guard row on each side: the region's edge pixels read there (never part of what is stored)
  __shared__ float rxs[TVR * (TVR + 2)], rys[TVR * (TVR + 2)], xs[TVR * (TVR + 2)];
  pdl_trigger();
  pdl_wait();
  const int c = blockIdx.z, n = a.n, halo = a.k + a.last, side = TVR - 2 * halo;
  const int N = n * n;
  const int lx = threadIdx.x % TVR, ly = threadIdx.x / TVR, l = TVR + threadIdx.x;
  const int ix = blockIdx.x * side - halo + lx, iy = blockIdx.y * side - halo + ly;
  const float lo = a.lo[c], hi = a.hi[c], lam = a.lam, step = a.step;
  const bool in = ix >= 0 && ix < n && iy >= 0 && iy < n, has_x = ix < n - 1, has_y = iy < n - 1;
  const int i = in ? iy * n + ix : 0;
  const float z = reinterpret_cast<const float*>(a.z)[2 * i + c];
  float rx = 0.f, ry = 0.f, px = 0.f, py = 0.f;
  if (!a.first && in) {
    const float *r = a.rin + 2 * c * N, *p = a.pin + 2 * c * N;
    rx = r[i];
    ry = r[N + i];
    px = p[i];
    py = p[N + i];
  }
  rxs[l] = rx;
  rys[l] = ry;
  if (ly == 0) rxs[lx] = rys[lx] = rxs[l + TVR * TVR] = rys[l + TVR * TVR] = xs[l + TVR * TVR] = 0.f;
  __syncthreads();
  // P_C(z - lam D^T r)
  auto xat = [&]() { return fminf(fmaxf(z - lam * (((rxs[l - 1] - rx) - ry) + rys[l - TVR]), lo), hi); };
  for (int k = 0; k < a.k; ++k) {
    const float x0 = xat();
    xs[l] = x0;
    __syncthreads();
    const float dx = has_x ? xs[l + 1] - x0 : 0.f, dy = has_y ? xs[l + TVR] - x0 : 0.f;
    float qx = rx + step * dx, qy = ry + step * dy;
    const float nn = qx * qx + qy * qy;
    if (nn > 1.f) {  // else the norm is at most 1 and the projection changes nothing
      const float nrm = sqrtf(nn);
      qx /= nrm;
      qy /= nrm;
    }
    const float beta = a.last && k == a.k - 1 ? 0.f : a.beta[k];  // the output step reads p
    rx = in ? qx + beta * (qx - px) : 0.f;
    ry = in ? qy + beta * (qy - py) : 0.f;
    px = qx;
    py = qy;
    rxs[l] = rx;
    rys[l] = ry;
    __syncthreads();
  }
  if (!in || lx < halo || lx >= TVR - halo || ly < halo || ly >= TVR - halo) return;
  if (!a.last) {
    float *r = a.rout + 2 * c * N, *p = a.pout + 2 * c * N;
    r[i] = rx;
    r[N + i] = ry;
    p[i] = px;
    p[N + i] = py;
    return;
  }
  const float xo = xat();
  float* x = reinterpret_cast<float*>(a.x + i) + c;
  if (a.s_out) {  // fprev is read before x (x may alias it)
    float* s = reinterpret_cast<float*>(a.s_out + i) + c;
    const float* fp = reinterpret_cast<const float*>(a.fprev + i) + c;
    s[0] = xo + a.beta_mom * (xo - fp[0]);
    if (a.ncomp == 1) s[1] = 0.f + a.beta_mom * (0.f - fp[1]);
  }
  x[0] = xo;
  if (a.ncomp == 1) x[1] = 0.f;
}

// `iters` >= 1 iterations and the output in as few launches of at most TV_KMAX iterations as they take, shared
// out evenly (the output step widens the last launch's halo by one)
static cisor_status tv_blocks(cisor_ctx* c, const float2* z, float2* x, double lam, int iters, double lo, double hi,
                              double lo_im, double hi_im, int ncomp, const float2* f_prev, double beta_mom,
                              float2* s_out) {
  TvBlock a{};
  a.z = z;
  a.n = c->n;
  a.lam = (float)lam;
  a.step = (float)(1.0 / (8.0 * lam));
  a.lo[0] = (float)lo;
  a.hi[0] = (float)hi;
  a.lo[1] = (float)lo_im;
  a.hi[1] = (float)hi_im;
  a.ncomp = ncomp;
  a.x = x;
  a.fprev = f_prev;
  a.beta_mom = (float)beta_mom;
  a.s_out = s_out;
  float *rin = c->tv_r0, *rout = c->tv_r1, *pin = c->tv_p, *pout = c->tva0;
  const int launches = (iters + TV_KMAX - 1) / TV_KMAX;
  double t = 1.0;
  for (int l = 0, done = 0; l < launches; ++l) {
    a.k = (iters - done) / (launches - l);
    a.first = l == 0;
    a.last = l == launches - 1;
    for (int k = 0; k < a.k; ++k) {
      const double tn = (1.0 + sqrt(1.0 + 4.0 * t * t)) / 2.0;
      a.beta[k] = (float)((t - 1.0) / tn);
      t = tn;
    }
    a.rin = rin;
    a.pin = pin;
    a.rout = rout;
    a.pout = pout;
    const int side = TVR - 2 * (a.k + a.last), g = (c->n + side - 1) / side;
    CISOR_CUDA(launch_pdl(tv_block_kernel, dim3(g, g, ncomp), dim3(TVR * TVR), 0, c->stream, a));
    c->launches += 1;
    done += a.k;
    float* q = rin;
    rin = rout;
    rout = q;
    q = pin;
    pin = pout;
    pout = q;
  }
  return CISOR_OK;
}

// (D^T r) at voxel (iz, iy, ix) of an n^3 volume, for the forward difference with zero difference at the last index
__device__ __forceinline__ float dt3_at(const float* __restrict__ rx, const float* __restrict__ ry,
                                        const float* __restrict__ rz, int iz, int iy, int ix, int n) {
  const long long nn = (long long)n * n;
  const long long i = iz * nn + (long long)iy * n + ix;
  float v = 0.f;
  if (ix < n - 1) v -= rx[i];
  if (ix > 0) v += rx[i - 1];
  if (iy < n - 1) v -= ry[i];
  if (iy > 0) v += ry[i - n];
  if (iz < n - 1) v -= rz[i];
  if (iz > 0) v += rz[i - nn];
  return v;
}

__global__ void tv_iter3_kernel(const float* __restrict__ zp, const float* __restrict__ rin, float* __restrict__ rout,
                                float* __restrict__ p, int n, float lam, float step, float beta, float lo0, float hi0,
                                float lo1, float hi1) {
  const int ix = blockIdx.x * blockDim.x + threadIdx.x;
  const int iy = blockIdx.y, iz = blockIdx.z % n, c = blockIdx.z / n;
  const long long nn = (long long)n * n, N = nn * n;
  const float lo = c ? lo1 : lo0, hi = c ? hi1 : hi0;
  const float* z = zp + c * N;
  const float* rx = rin + 3 * c * N;
  const float* ry = rx + N;
  const float* rz = ry + N;
  const bool valid = ix < n;
  const int xi = valid ? ix : n - 1;
  const long long i = iz * nn + (long long)iy * n + xi;
  auto xat = [&](int zz, int yy, int xx, long long j) {
    return fminf(fmaxf(z[j] - lam * dt3_at(rx, ry, rz, zz, yy, xx, n), lo), hi);
  };
  const float x0 = xat(iz, iy, xi, i);
  // right neighbour from the next lane; the last lane of a warp computes it itself
  float xr = __shfl_down_sync(0xffffffffu, x0, 1);
  const int lane = threadIdx.x & 31;
  if (lane == 31 && xi < n - 1) xr = xat(iz, iy, xi + 1, i + 1);
  if (!valid) return;
  const float dx = (ix < n - 1) ? xr - x0 : 0.f;
  const float dy = (iy < n - 1) ? xat(iz, iy + 1, ix, i + n) - x0 : 0.f;
  const float dz = (iz < n - 1) ? xat(iz + 1, iy, ix, i + nn) - x0 : 0.f;
  const float qx = rx[i] + step * dx, qy = ry[i] + step * dy, qz = rz[i] + step * dz;
  const float nrm = fmaxf(1.f, sqrtf(qx * qx + qy * qy + qz * qz));
  const float px = qx / nrm, py = qy / nrm, pz = qz / nrm;
  float* pc = p + 3 * c * N;
  const float pox = pc[i], poy = pc[N + i], poz = pc[2 * N + i];
  pc[i] = px;
  pc[N + i] = py;
  pc[2 * N + i] = pz;
  float* ro = rout + 3 * c * N;
  ro[i] = px + beta * (px - pox);
  ro[N + i] = py + beta * (py - poy);
  ro[2 * N + i] = pz + beta * (pz - poz);
}

// x = P_C(z - lam D^T p) of a volume, or the clamp of N values where lam = 0, and the momentum
__global__ void tv_final_kernel(const float* __restrict__ zp, const float* __restrict__ p, int n, long long N, float lam,
                                float lo0, float hi0, float lo1, float hi1, int ncomp, float2* x, const float2* fprev,
                                float beta_mom, float2* __restrict__ s_out) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int ix = (int)(i % n), iy = (int)((i / n) % n), iz = (int)(i / ((long long)n * n));
  float xv[2] = {0.f, 0.f};
  for (int c = 0; c < ncomp; ++c) {
    const float lo = c ? lo1 : lo0, hi = c ? hi1 : hi0;
    const float* pc = p + 3 * c * N;
    const float d = lam > 0.f ? dt3_at(pc, pc + N, pc + 2 * N, iz, iy, ix, n) : 0.f;
    xv[c] = fminf(fmaxf(zp[c * N + i] - lam * d, lo), hi);
  }
  const float2 xo = make_float2(xv[0], xv[1]);
  if (s_out) {
    const float2 fp = fprev[i];  // read before x (x may alias fprev)
    s_out[i] = make_float2(xo.x + beta_mom * (xo.x - fp.x), xo.y + beta_mom * (xo.y - fp.y));
  }
  x[i] = xo;
}

// z_j = z for every piece j of every plane: layout (plane * m + j) * N
__global__ void tv_ppa_init_kernel(const float2* __restrict__ z, float* __restrict__ zs, long long N, int m,
                                   int ncomp) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const float2 v = z[i];
  for (int c = 0; c < ncomp; ++c)
    for (int j = 0; j < m; ++j) zs[((long long)c * m + j) * N + i] = c ? v.y : v.x;
}

__device__ __forceinline__ float soft(float d, float t) { return copysignf(fmaxf(fabsf(d) - t, 0.f), d); }

template <int D>
__global__ void __launch_bounds__(256) tv_ppa_kernel(const float* __restrict__ zin, float* __restrict__ zout, int n,
                                                     float cthr, float lo0, float hi0, float lo1, float hi1, int ncomp,
                                                     int last, float2* x_out, const float2* fprev, float beta_mom,
                                                     float2* __restrict__ s_out) {
  constexpr int M = 2 * D + 1;
  const long long nn = (long long)n * n;
  const long long N = D == 3 ? nn * n : nn;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int coord[3] = {(int)(i % n), (int)((i / n) % n), (int)(i / nn)};
  const long long stride[3] = {1, n, nn};
  float xv[2] = {0.f, 0.f};
  for (int c = 0; c < ncomp; ++c) {
    const float* zc = zin + (long long)c * M * N;
    float zj[M], p[M];
    float acc = 0.f;
#pragma unroll
    for (int j = 0; j < 2 * D; ++j) {
      const int a = j >> 1, par = j & 1, pos = coord[a];
      const float* zp = zc + (long long)j * N;
      const float v = zp[i];
      zj[j] = v;
      const int rel = pos - par;
      float pj = v;
      if (rel >= 0 && (rel & 1) == 0 && pos + 1 < n) {  // first of the pair (pos, pos + 1)
        const float w = zp[i + stride[a]];
        pj = 0.5f * (v + w) - 0.5f * soft(w - v, 2.f * cthr);
      } else if (rel >= 1 && (rel & 1) == 1) {          // second of the pair (pos - 1, pos)
        const float w = zp[i - stride[a]];
        pj = 0.5f * (w + v) + 0.5f * soft(v - w, 2.f * cthr);
      }
      p[j] = pj;
      acc += pj;
    }
    const float lo = c ? lo1 : lo0, hi = c ? hi1 : hi0;
    zj[2 * D] = zc[(long long)(2 * D) * N + i];
    p[2 * D] = fminf(fmaxf(zj[2 * D], lo), hi);
    acc += p[2 * D];
    const float x = acc * (1.f / M);
    xv[c] = x;
    if (!last) {
      float* zo = zout + (long long)c * M * N;
#pragma unroll
      for (int j = 0; j < M; ++j) zo[(long long)j * N + i] = x + zj[j] - p[j];
    }
  }
  if (last) {
    const float2 xo = make_float2(xv[0], xv[1]);
    if (s_out) {
      const float2 fp = fprev[i];  // read before x (x may alias fprev)
      s_out[i] = make_float2(xo.x + beta_mom * (xo.x - fp.x), xo.y + beta_mom * (xo.y - fp.y));
    }
    x_out[i] = xo;
  }
}

cisor_status tv_prox_aniso(cisor_ctx* c, const float2* z, float2* x, double lam, int iters, double lo, double hi,
                           double lo_im, double hi_im, int complex_f, const float2* f_prev, double beta_mom,
                           float2* s_out) {
  if (!(lam > 0.0) || iters < 1)  // the prox of the box alone is the clamp (the FGP path's last kernel)
    return tv_prox(c, z, x, 0.0, 0, lo, hi, lo_im, hi_im, complex_f, f_prev, beta_mom, s_out);
  const long long N = c->N;
  const int ncomp = complex_f ? 2 : 1;
  const int m = 2 * c->dim + 1;
  const unsigned gN = (unsigned)((N + 255) / 256);
  tv_ppa_init_kernel<<<gN, 256, 0, c->stream>>>(z, c->tva0, N, m, ncomp);
  CISOR_CUDA(cudaGetLastError());
  c->launches += 1;
  float* zin = c->tva0;
  float* zout = c->tva1;
  const float cthr = (float)(m * lam);
  for (int k = 0; k < iters; ++k) {
    const int last = k == iters - 1;
    if (c->dim == 3)
      tv_ppa_kernel<3><<<gN, 256, 0, c->stream>>>(zin, zout, c->n, cthr, (float)lo, (float)hi, (float)lo_im,
                                                  (float)hi_im, ncomp, last, x, f_prev, (float)beta_mom, s_out);
    else
      tv_ppa_kernel<2><<<gN, 256, 0, c->stream>>>(zin, zout, c->n, cthr, (float)lo, (float)hi, (float)lo_im,
                                                  (float)hi_im, ncomp, last, x, f_prev, (float)beta_mom, s_out);
    CISOR_CUDA(cudaGetLastError());
    c->launches += 1;
    float* t = zin;
    zin = zout;
    zout = t;
  }
  return CISOR_OK;
}

cisor_status tv_prox(cisor_ctx* c, const float2* z, float2* x, double lam, int iters, double lo, double hi,
                     double lo_im, double hi_im, int complex_f, const float2* f_prev, double beta_mom,
                     float2* s_out) {
  const int n = c->n;
  const long long N = c->N;
  const int ncomp = complex_f ? 2 : 1;
  const unsigned gN = (unsigned)((N + 255) / 256);
  const bool tv = lam > 0.0 && iters > 0;  // else the clamp
  if (c->dim == 2 && tv)
    return tv_blocks(c, z, x, lam, iters, lo, hi, lo_im, hi_im, ncomp, f_prev, beta_mom, s_out);
  tv_split_kernel<<<gN, 256, 0, c->stream>>>(z, c->tv_z, tv ? c->tv_r0 : nullptr, c->tv_p, N, ncomp);
  CISOR_CUDA(cudaGetLastError());
  c->launches += 1;
  if (tv) {
    const int bx = ((n + 31) / 32) * 32 > 256 ? 256 : ((n + 31) / 32) * 32;
    dim3 g((n + bx - 1) / bx, n, n * ncomp);
    double t = 1.0;
    float* rin = c->tv_r0;
    float* rout = c->tv_r1;
    const float step = (float)(1.0 / (12.0 * lam));
    for (int k = 0; k < iters; ++k) {
      const double tn = (1.0 + sqrt(1.0 + 4.0 * t * t)) / 2.0;
      const float beta = (float)((t - 1.0) / tn);
      tv_iter3_kernel<<<g, bx, 0, c->stream>>>(c->tv_z, rin, rout, c->tv_p, n, (float)lam, step, beta, (float)lo,
                                               (float)hi, (float)lo_im, (float)hi_im);
      CISOR_CUDA(cudaGetLastError());
      c->launches += 1;
      float* tmp = rin;
      rin = rout;
      rout = tmp;
      t = tn;
    }
  }
  tv_final_kernel<<<gN, 256, 0, c->stream>>>(c->tv_z, c->tv_p, n, N, tv ? (float)lam : 0.f, (float)lo, (float)hi, (float)lo_im,
                                             (float)hi_im, ncomp, x, f_prev, (float)beta_mom, s_out);
  CISOR_CUDA(cudaGetLastError());
  c->launches += 1;
  return CISOR_OK;
}

}  // namespace cisor
