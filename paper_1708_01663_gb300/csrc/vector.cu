// The 3D vectorial model of the appendix ("3D Diffractive Imaging").
//
// Fields are E = (E^(1), E^(2), E^(3)) stored [T, 3, N] (component-major per
// transmitter), so the three components of a transmitter are three
// consecutive transforms of the scalar FFT convolution (ConvOp::tx_div = 3).
// With C = k^2 B = conv_G(f E) (G the k^2-weighted scalar matrix of Eq. 3, so
// B = G~ (f E) of the appendix):
//     A x   = x - C - D C / k^2                        (discrete constraint)
//     A^H x = x - conj(f) conv_{G^H}(x + D x / k^2)    (D real and symmetric)
// D is the appendix's finite-difference grad-div operator: the 3-point second
// difference for d^2/dx_c^2 and the 4-point diagonal stencil / (4 delta^2)
// for the mixed derivatives, acting on grid values only (neighbours outside
// the grid count as zero).  The forward matvec runs the stencil as the
// epilogue of the convolution (A x, b - A x and the dot slots of the Krylov
// solver); the adjoint runs it before the convolution, whose inverse-row
// epilogue then forms the result.  Dot partials of both land in the
// [T][3 nblk][DOT_SLOTS] slots that the solver's scalar step sums: the adjoint's
// as nblk per component, the forward's one per CTA over all components with
// zeros in the slots behind them.
//
// Tables: H~ [M, 3N] = delta^3 times row 3 of the dyadic Green's function
//     G(r) = k^2 [ (3/(kd)^2 - 3j/(kd) - 1) r^ r^T + (1 + j/(kd) - 1/(kd)^2) I ] g(d)
// (the receivers measure the z component), and polarised plane waves
// E_in,t = p_t exp(j k d_t . r).
#include <math.h>

#include "common.cuh"
#include "dots.cuh"

namespace cisor {

// besides the inner products (DOTS_NONE .. DOTS_ANY) of an A x pass: the adjoint's pre-pass
enum { VEC_PRE = -1 };

struct VecEpiArgs {
  const float2* C;      // conv output [ntx, 3, N] (forward) or the field x (pre-pass)
  const float2* x;      // the x of A x
  const float2* aux;
  float2* out;
  float2* out2;
  int epi;              // EPI_MATVEC, EPI_RESID; VEC_PRE: pre-pass w = x + D x / k^2
  int need_aux;
  int dot_a[DOT_SLOTS], dot_b[DOT_SLOTS];
  const int* active;
  float* part;
  int n, nblk;
  long long N;
  float inv_k2, inv_d2;
};

constexpr int VS_Z = 4;  // output planes per CTA (of 4, 8, 16: 8 is 1% faster at 32^3, 4 by 8% at 16^3)

// All three components of 256 (x, y) columns over VS_Z planes of transmitter blockIdx.z; a thread marches along z.
// The mixed derivatives along z are differences over z of in-plane differences,
//     (D F)^(x) ~ M0(z + 1) - M0(z - 1),  M0 = F2(x + 1) - F2(x - 1)   (1 / 4 delta^2; y likewise, z from F0 and F1),
// so a plane's values are read once and kept as M0, M1, M2 and the centre of F2 for the three planes they act on: 19
// reads a voxel for the three components instead of 33, one set of bounds tests, and no component's field read by
// three CTAs (one component a CTA took 15 plane reads through L2 for the 3 it needs).  Bound by memory: C, x and the
// result are 64 MB each at 81 transmitters, 32^3, 28 us at the copy rate.  There a pass fell from 65 us to 36 (A x) and
// 41 (pre-pass), A x as a whole from 315 to 287, A^H x from 302 to 279; with 16 transmitters 68 to 64 and 66 to 60.
// Three CTAs an SM (80 registers): two hide less (293 / 289), four spill (310 / 301).
// The solver's sets of inner products are compiled in (dots.cuh; a pass with them 53 us by operand codes, the gradient
// of 81 transmitters 8.09 -> 7.96 ms).
template <int DK>
__global__ void __launch_bounds__(256, 3) vec_stencil_kernel(const VecEpiArgs a) {
  const int t = blockIdx.z;
  if (a.active && !a.active[t]) return;
  const int N = (int)a.N, n = a.n, n2 = n * n;
  const int col = blockIdx.x * 256 + threadIdx.x, z0 = blockIdx.y * VS_Z, z1 = min(n, z0 + VS_Z);
  const long long base = (long long)t * 3 * N;
  float2 acc[DOT_SLOTS];
#pragma unroll
  for (int s = 0; s < DOT_SLOTS; ++s) acc[s] = make_float2(0.f, 0.f);
  if (col < n2) {
    const int iy = col / n, ix = col - iy * n;
    const bool xl = ix > 0, xr = ix < n - 1, yl = iy > 0, yr = iy < n - 1;
    const float2* F0 = a.C + base + (long long)z0 * n2 + col;  // plane z0; planes z0 - 1 .. z1 by offset
    const float2 *F1 = F0 + N, *F2 = F1 + N;
    const float2 zero = make_float2(0.f, 0.f);
    auto at = [&](const float2* p, int o, bool in) { return in ? __ldg(p + o) : zero; };
    const float q = 0.25f * a.inv_d2;
    // of the plane before, this one and the next
    float2 m0[3], m1[3], m2[3], c2[3], c0, c1, d0, d1;
    auto load = [&](int z, float2& M0, float2& M1, float2& M2, float2& C2, float2& C0, float2& C1, float2& D0, float2& D1) {
      const bool in = z >= 0 && z < n;
      const int o = (z - z0) * n2;
      const bool l = in && xl, r = in && xr, b = in && yl, u = in && yr;
      const float2 e0 = at(F0, o - 1, l), e1 = at(F0, o + 1, r), g0 = at(F1, o - n, b), g1 = at(F1, o + n, u);
      C0 = at(F0, o, in);
      C1 = at(F1, o, in);
      C2 = at(F2, o, in);
      M0 = c_sub(at(F2, o + 1, r), at(F2, o - 1, l));
      M1 = c_sub(at(F2, o + n, u), at(F2, o - n, b));
      M2 = c_add(c_sub(e1, e0), c_sub(g1, g0));
      if (z >= z0 && z < z1) {  // the in-plane parts of components x and y
        D0 = c_add(c_scale(c_add(c_scale(C0, -2.f), c_add(e0, e1)), a.inv_d2),
                   c_scale(c_sub(c_sub(at(F1, o + 1 + n, r && u), at(F1, o + 1 - n, r && b)),
                                 c_sub(at(F1, o - 1 + n, l && u), at(F1, o - 1 - n, l && b))), q));
        D1 = c_add(c_scale(c_add(c_scale(C1, -2.f), c_add(g0, g1)), a.inv_d2),
                   c_scale(c_sub(c_sub(at(F0, o + 1 + n, r && u), at(F0, o + 1 - n, r && b)),
                                 c_sub(at(F0, o - 1 + n, l && u), at(F0, o - 1 - n, l && b))), q));
      }
    };
    float2 n0, n1, nd0, nd1;
    load(z0 - 1, m0[0], m1[0], m2[0], c2[0], n0, n1, nd0, nd1);
    load(z0, m0[1], m1[1], m2[1], c2[1], c0, c1, d0, d1);
    constexpr int UN = DK > DOTS_NONE ? 1 : 2;  // (inner products leave no registers for two planes)
#pragma unroll UN
    for (int z = z0; z < z1; ++z) {
      const long long i0 = base + (long long)z * n2 + col;
      float2 xv[3], av[3];  // (read before the stores, which the compiler must take for aliases)
      if (DK != VEC_PRE) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          xv[c] = a.x[i0 + (long long)c * N];
          av[c] = DK == DOTS_RV || DK == DOTS_RES || a.need_aux ? a.aux[i0 + (long long)c * N] : zero;
        }
      }
      load(z + 1, m0[2], m1[2], m2[2], c2[2], n0, n1, nd0, nd1);
      const float2 dc[3] = {c_add(d0, c_scale(c_sub(m0[2], m0[0]), q)), c_add(d1, c_scale(c_sub(m1[2], m1[0]), q)),
                            c_add(c_scale(c_add(c_scale(c2[1], -2.f), c_add(c2[0], c2[2])), a.inv_d2),
                                  c_scale(c_sub(m2[2], m2[0]), q))};
      const float2 ctr[3] = {c0, c1, c2[1]};
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const long long idx = i0 + (long long)c * N;
        if (DK == VEC_PRE) {  // pre-pass of the adjoint: w = x + D x / k^2
          a.out[idx] = c_add(ctr[c], c_scale(dc[c], a.inv_k2));
        } else {
          float2 y = c_sub(c_sub(xv[c], ctr[c]), c_scale(dc[c], a.inv_k2));
          if (a.epi == EPI_RESID) y = c_sub(av[c], y);
          a.out[idx] = y;
          if (a.out2) a.out2[idx] = y;
          if constexpr (DK > DOTS_NONE && DK < DOTS_ANY) {
            dots_accumulate<DK>(ConvOp{}, acc, y, xv[c], av[c]);  // (fixed operands: the codes are not read)
          } else if constexpr (DK == DOTS_ANY) {
#pragma unroll
            for (int s = 0; s < DOT_SLOTS; ++s)
              if (a.dot_a[s]) acc[s] = c_add(acc[s], c_cjmul(pick(a.dot_a[s], y, xv[c], av[c]), pick(a.dot_b[s], y, xv[c], av[c])));
          }
        }
      }
      m0[0] = m0[1], m1[0] = m1[1], m2[0] = m2[1], c2[0] = c2[1];
      m0[1] = m0[2], m1[1] = m1[2], m2[1] = m2[2], c2[1] = c2[2];
      c0 = n0, c1 = n1, d0 = nd0, d1 = nd1;
    }
  }
  if constexpr (DK > DOTS_NONE) {  // a partial per CTA, zeros in the other slots of the transmitter's 3 nblk
    float2* part = reinterpret_cast<float2*>(a.part) + (size_t)t * 3 * a.nblk * DOT_SLOTS;
    const int cta = blockIdx.y * gridDim.x + blockIdx.x, ctas = gridDim.x * gridDim.y;
    block_dots<256, DotSlots<DK>::MASK>(acc, part + (size_t)cta * DOT_SLOTS);
    for (int b = cta + ctas; b < 3 * a.nblk; b += ctas)
      if (threadIdx.x < DOT_SLOTS) part[(size_t)b * DOT_SLOTS + threadIdx.x] = make_float2(0.f, 0.f);
  }
}

static VecEpiArgs stencil_args(cisor_ctx* c) {
  VecEpiArgs a{};
  a.n = c->n;
  a.N = c->N;
  a.nblk = c->nblk;
  a.part = c->part;
  a.inv_k2 = (float)(1.0 / (c->k * c->k));
  a.inv_d2 = (float)(1.0 / (c->delta * c->delta));
  return a;
}

static cisor_status launch_stencil(cisor_ctx* c, const VecEpiArgs& a, int ntx) {
  // (at most 3 nblk CTAs a transmitter, the slots of its partials: nblk is n^2 / 32 or more)
  const dim3 g((unsigned)((c->n * c->n + 255) / 256), (unsigned)((c->n + VS_Z - 1) / VS_Z), ntx);
  ConvOp dots{};
  for (int k = 0; k < DOT_SLOTS; ++k) {
    dots.dot_a[k] = a.dot_a[k];
    dots.dot_b[k] = a.dot_b[k];
  }
  switch (a.epi == VEC_PRE ? (int)VEC_PRE : dots_kind(dots)) {
    case VEC_PRE: vec_stencil_kernel<VEC_PRE><<<g, 256, 0, c->stream>>>(a); break;
    case DOTS_NONE: vec_stencil_kernel<DOTS_NONE><<<g, 256, 0, c->stream>>>(a); break;
    case DOTS_RV: vec_stencil_kernel<DOTS_RV><<<g, 256, 0, c->stream>>>(a); break;
    case DOTS_TS: vec_stencil_kernel<DOTS_TS><<<g, 256, 0, c->stream>>>(a); break;
    case DOTS_RES: vec_stencil_kernel<DOTS_RES><<<g, 256, 0, c->stream>>>(a); break;
    default: vec_stencil_kernel<DOTS_ANY><<<g, 256, 0, c->stream>>>(a);
  }
  CISOR_CUDA(cudaGetLastError());
  c->launches += 1;
  return CISOR_OK;
}

cisor_status vec_matvec(cisor_ctx* c, const VecOp& op) {
  if (!op.adjoint) {
    ConvOp co{};
    co.mul_f = 1;
    co.prologue = PRO_COPY;
    co.src = op.x;
    co.epilogue = EPI_CONV_ADD;
    co.out = c->vbuf;
    co.f = op.f;
    co.ntx = 3 * op.ntx;
    co.tx_div = 3;
    co.active = op.active;
    CISOR_TRY(conv_pass(c, co));
    VecEpiArgs a = stencil_args(c);
    a.C = c->vbuf;
    a.x = op.x;
    a.aux = op.aux;
    a.out = op.out;
    a.out2 = op.out2;
    a.epi = op.epilogue;
    for (int s = 0; s < DOT_SLOTS; ++s) {
      a.dot_a[s] = op.dot_a[s];
      a.dot_b[s] = op.dot_b[s];
    }
    a.need_aux = op.epilogue == EPI_RESID;
    for (int s = 0; s < DOT_SLOTS; ++s) a.need_aux |= op.dot_a[s] == OP_AUX || op.dot_b[s] == OP_AUX;
    a.active = op.active;
    return launch_stencil(c, a, op.ntx);
  }
  VecEpiArgs a = stencil_args(c);
  a.C = op.x;
  a.out = c->vbuf;
  a.epi = VEC_PRE;
  a.active = op.active;
  CISOR_TRY(launch_stencil(c, a, op.ntx));
  ConvOp co{};
  co.adjoint = 1;
  co.mul_f = 1;
  co.prologue = PRO_COPY;
  co.src = c->vbuf;
  co.epilogue = op.epilogue;
  co.esrc = op.x;
  co.aux = op.aux;
  co.out = op.out;
  co.out2 = op.out2;
  co.gz = op.gz;
  co.zadd = op.zadd;
  for (int s = 0; s < DOT_SLOTS; ++s) {
    co.dot_a[s] = op.dot_a[s];
    co.dot_b[s] = op.dot_b[s];
  }
  co.part = c->part;
  co.f = op.f;
  co.ntx = 3 * op.ntx;
  co.tx_div = 3;
  co.active = op.active;
  return conv_pass(c, co);
}

cisor_status vec_gz(cisor_ctx* c) {
  VecEpiArgs a = stencil_args(c);
  a.C = c->vadj;
  a.out = c->vbuf;
  a.epi = VEC_PRE;
  CISOR_TRY(launch_stencil(c, a, c->T));
  ConvOp co{};
  co.adjoint = 1;
  co.prologue = PRO_COPY;
  co.src = c->vbuf;
  co.epilogue = EPI_CONV_ADD;
  co.aux = c->z;
  co.out = c->gz;
  co.f = c->f;
  co.ntx = 3 * c->T;
  co.tx_div = 3;
  return conv_pass(c, co);
}

// p = r + beta (p - omega v) (p = r when beta = 0) and s = r - alpha v over [ntx, Nf]
__global__ void __launch_bounds__(256) vec_pupdate_kernel(long long Nf, const int* __restrict__ active,
                                                          const double* __restrict__ scal, const float2* __restrict__ r,
                                                          float2* __restrict__ p, const float2* __restrict__ v) {
  const int t = blockIdx.y;
  if (!active[t]) return;
  const double2* sc = reinterpret_cast<const double2*>(scal) + (size_t)t * SC_STRIDE;
  const float2 beta = z_to_c(sc[SC_BETA]), omega = z_to_c(sc[SC_OMEGA]);
  const bool fresh = beta.x == 0.f && beta.y == 0.f;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < Nf; i += (long long)gridDim.x * blockDim.x) {
    const long long k = (long long)t * Nf + i;
    p[k] = fresh ? r[k] : c_add(r[k], c_mul(beta, c_sub(p[k], c_mul(omega, v[k]))));
  }
}

__global__ void __launch_bounds__(256) vec_axpy_kernel(long long Nf, const int* __restrict__ active,
                                                       const double* __restrict__ scal, const float2* __restrict__ r,
                                                       const float2* __restrict__ v, float2* __restrict__ s) {
  const int t = blockIdx.y;
  if (!active[t]) return;
  const float2 alpha = z_to_c(reinterpret_cast<const double2*>(scal)[(size_t)t * SC_STRIDE + SC_ALPHA]);
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < Nf; i += (long long)gridDim.x * blockDim.x) {
    const long long k = (long long)t * Nf + i;
    s[k] = c_sub(r[k], c_mul(alpha, v[k]));
  }
}

static unsigned vec_blocks(long long Nf) {
  const long long b = (Nf + 1023) / 1024;
  return (unsigned)(b < 1 ? 1 : b);
}

cisor_status vec_pupdate(cisor_ctx* c, int ntx) {
  vec_pupdate_kernel<<<dim3(vec_blocks(c->Nf), ntx), 256, 0, c->stream>>>(c->Nf, c->active, c->scal, c->r, c->p, c->v);
  CISOR_CUDA(cudaGetLastError());
  c->launches += 1;
  return CISOR_OK;
}

cisor_status vec_axpy(cisor_ctx* c, int ntx) {
  vec_axpy_kernel<<<dim3(vec_blocks(c->Nf), ntx), 256, 0, c->stream>>>(c->Nf, c->active, c->scal, c->r, c->v, c->s);
  CISOR_CUDA(cudaGetLastError());
  c->launches += 1;
  return CISOR_OK;
}

// ---------------------------------------------------------------- tables (FP64)
__global__ void dyadic_sensing_kernel(const SenseTable H, const double* rx, int M, int n, double delta, double k) {
  const long long N = (long long)n * n * n, K = 3 * N;
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)M * K) return;
  const int m = (int)(idx / K);
  const long long rem = idx % K;
  const int c = (int)(rem / N);
  const long long p = rem % N;
  const double h = n / 2.0 - 0.5;
  const double dx = rx[3 * m] - ((int)(p % n) - h) * delta;
  const double dy = rx[3 * m + 1] - ((int)((p / n) % n) - h) * delta;
  const double dz = rx[3 * m + 2] - ((int)(p / ((long long)n * n)) - h) * delta;
  const double d = sqrt(dx * dx + dy * dy + dz * dz);
  const double rh[3] = {dx / d, dy / d, dz / d};
  const double kd = k * d;
  double sn, cs;
  sincos(kd, &sn, &cs);
  const double2 g = make_double2(cs / (4.0 * 3.14159265358979323846 * d), sn / (4.0 * 3.14159265358979323846 * d));
  // a = 3/(kd)^2 - 1 - 3j/(kd), b = 1 - 1/(kd)^2 + j/(kd)
  const double2 av = make_double2(3.0 / (kd * kd) - 1.0, -3.0 / kd);
  const double2 bv = make_double2(1.0 - 1.0 / (kd * kd), 1.0 / kd);
  double2 coef = make_double2(av.x * rh[2] * rh[c], av.y * rh[2] * rh[c]);
  if (c == 2) coef = z_add(coef, bv);
  const double s = k * k * delta * delta * delta;
  const double2 v = z_mul(coef, g);
  H.store(m, rem, make_float2((float)(s * v.x), (float)(s * v.y)));
}

__global__ void polarised_wave_kernel(float2* u, const double* tx, int T, int n, double delta, double k) {
  const long long N = (long long)n * n * n;
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)T * 3 * N) return;
  const int t = (int)(idx / (3 * N));
  const long long rem = idx % (3 * N);
  const int c = (int)(rem / N);
  const long long p = rem % N;
  const double h = n / 2.0 - 0.5;
  const double* d = tx + 6 * t;
  const double ph = k * delta * (d[0] * ((int)(p % n) - h) + d[1] * ((int)((p / n) % n) - h) +
                                 d[2] * ((int)(p / ((long long)n * n)) - h));
  double sn, cs;
  sincos(ph, &sn, &cs);
  const double pol = d[3 + c];
  u[idx] = make_float2((float)(pol * cs), (float)(pol * sn));
}

cisor_status vec_tables(cisor_ctx* c, const double* d_tx, const double* d_rx) {
  const long long MK = (long long)c->M * c->Nf, TK = (long long)c->T * c->Nf;
  dyadic_sensing_kernel<<<(unsigned)((MK + 255) / 256), 256, 0, c->stream>>>(sense_table(c), d_rx, c->M, c->n, c->delta, c->k);
  CISOR_CUDA(cudaGetLastError());
  polarised_wave_kernel<<<(unsigned)((TK + 255) / 256), 256, 0, c->stream>>>(c->u_in, d_tx, c->T, c->n, c->delta, c->k);
  CISOR_CUDA(cudaGetLastError());
  return CISOR_OK;
}

}  // namespace cisor
