// Batched 3D FFT convolution for P = 64 and 128 as three kernels (Sec. II,
// Eqs. 3-4), the 3D counterpart of conv.cu's 2D pass with the same prologues,
// epilogues and inner products:
//
//  1. conv3_rows_fwd : prologue, times f, FFT along x of RB3 x rows; the row
//                      spectra go to R [T][kx][z][y], so that
//  2. conv3_plane    : one CTA takes the whole (z, y) plane of one x frequency
//                      of one transform: FFT along y and z, ghat product,
//                      inverse along z and y, n x n values in, n x n out, with
//                      the n x P half-transformed plane in shared memory.
//  3. conv3_rows_inv : inverse FFT along x, crop, epilogue and dot products.
//
// Why planes: five kernels (rows, y, z with ghat, y back, rows back) passed the
// padded intermediate through HBM five times, growing it to n P^2 values
// between the y and z kernels: 2.4 GB a pass at 48 transforms of n = 64, P =
// 128.  Here it never leaves n^2 P values and moves twice (0.8 GB); a plane's
// 64 KB and the 32 KB of its column exchanges leave room for two CTAs an SM.  Measured, one pass:
// 48 transforms of n = 64 554 -> 465 us (two-stage column kernels before), 243
// of n = 32 (81 vectorial fields, with their stencil) 400 -> 305 us, 20 of n = 40
// 223 -> 130 us; no size measured is slower.  The plane kernel (69 %
// of a pass of eight transforms of n = 64) is bound by shared-memory traffic (its
// pipe 72 % busy, issue 60 %, FMA pipe 45 %, DRAM 8 %): the two exchanges and the
// passes over the plane between the directions.
//
// Transforms are two-stage, P = E x 8 (128 = 16 x 8, 64 = 8 x 8): E elements a
// thread, 8 threads a transform, one exchange each way, arranged as
// conv_cols_2s does (radix E, then 8; back: radix 8 on the registers in place,
// then E).  A warp holds four transforms and every exchange of the plane kernel
// stays inside the warp (__syncwarp); the CTA meets only between the y and z
// directions.  plane_layout.cuh has the shared-memory layout: no access of a
// half-warp meets a bank twice (enumerated in tests/test_plane_layout.py).  A
// column has only P / 2 slots of its own in the plane; its exchange puts the
// other half into xs.
//
// ghat of a cubic grid depends only on |k| per axis and is the same under any
// permutation of the axes, so one eighth of it is kept in the order in which the
// plane kernel reads it (plane_ghat_kernel).
#include "common.cuh"
#include "dots.cuh"
#include "fft.cuh"
#include "plane_layout.cuh"
#include "regfft.cuh"

namespace cisor {

template <int P> struct Plane : PlaneLayout<P> {
  static constexpr int MINB = P == 128 ? 2 : 4;  // resident CTAs of the plane kernel per SM
};

// tw[r j] in the layout of PlaneLayout::tw
template <int P>
__device__ __forceinline__ void plane_twiddles(float2* t, const float2* __restrict__ tw, int nthr) {
  constexpr int E = Plane<P>::E, NT = Plane<P>::NT;
  for (int i = threadIdx.x; i < NT * E; i += nthr) t[Plane<P>::tw(i / E, i % E)] = tw[(i / E) * (i % E)];
}

// forward radix-8 stage of the exchanged elements x(q, r) (element j + E r, j = lt + 8 q) into v[8 q + r']
template <int P, class X>
__device__ __forceinline__ void plane_fwd8(float2* v, const float2* t, int lt, X x) {
  constexpr int NT = Plane<P>::NT, Q = Plane<P>::Q;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
#pragma unroll
    for (int r = 0; r < NT; ++r) {
      const float2 a = x(q, r);
      v[NT * q + r] = r == 0 ? a : c_mul(a, t[Plane<P>::tw(r, lt + NT * q)]);
    }
    dft8<false, true>(v + NT * q);
  }
}

// inverse radix-E stage of the exchanged elements x(r) (element lt + 8 r)
template <int P, class X>
__device__ __forceinline__ void plane_invE(float2* v, const float2* t, int lt, X x) {
  constexpr int E = Plane<P>::E;
#pragma unroll
  for (int r = 0; r < E; ++r) {
    const float2 a = x(r);
    v[r] = r == 0 ? a : c_mulcj(a, t[Plane<P>::tw(lt, r)]);
  }
  dft_n<E, true>(v);
}

// Rows kernels: RB3 rows of 8 threads per 256-thread CTA.
constexpr int RB3 = 32;

template <int P, int PRO>
__global__ void __launch_bounds__(256) conv3_rows_fwd(const ConvOp op, const float2* __restrict__ tw_g,
                                                      float2* __restrict__ R, int n, int nrows) {
  typedef Plane<P> PL;
  constexpr int E = PL::E, NT = PL::NT, Q = PL::Q;
  __shared__ float2 tw[PL::TW];
  __shared__ __align__(16) unsigned char buf[P * RB3 * 8];
  pdl_trigger();
  pdl_wait();
  const int tx = op.tx0 + blockIdx.y;
  const int txs = op.tx_div > 1 ? tx / op.tx_div : tx;
  if (op.active && !op.active[txs]) return;
  plane_twiddles<P>(tw, tw_g, 256);
  const int lt = threadIdx.x % NT, row = threadIdx.x / NT;
  const int iq = blockIdx.x * RB3 + row;
  const bool rowok = iq < nrows;
  float2 alpha = make_float2(0.f, 0.f), beta = alpha, omega = alpha;
  if (PRO != PRO_COPY) {
    const double2* sc = reinterpret_cast<const double2*>(op.scal) + (size_t)txs * SC_STRIDE;
    alpha = z_to_c(sc[SC_ALPHA]);
    beta = z_to_c(sc[SC_BETA]);
    omega = z_to_c(sc[SC_OMEGA]);
  }
  const bool mulf = op.mul_f && !op.adjoint;
  const bool fresh = (beta.x == 0.f && beta.y == 0.f);  // beta = 0 starts (or restarts) with p = r
  const long long row0 = (long long)iq * n, base = (long long)tx * nrows * n + row0;
  float2 v[E];
#pragma unroll
  for (int r = 0; r < E / 2; ++r) {  // n <= P/2: the upper half is padding
    const int ix = lt + NT * r;
    float2 val = make_float2(0.f, 0.f);
    if (rowok && ix < n) {
      const long long idx = base + ix;
      if (PRO == PRO_COPY) {
        val = op.src[idx];
      } else if (PRO == PRO_PUPDATE) {
        const float2 rv = op.src[idx];
        float2 p = rv;
        if (!fresh) p = c_add(rv, c_mul(beta, c_sub(op.pvec[idx], c_mul(omega, op.vvec[idx]))));
        op.pvec[idx] = p;
        val = p;
      } else {  // PRO_AXPY
        const float2 s = c_sub(op.src[idx], c_mul(alpha, op.vvec[idx]));
        op.svec[idx] = s;
        val = s;
      }
      if (mulf) val = c_mul(val, op.f[row0 + ix]);
    }
    v[r] = val;
  }
  dft_n_lo<E, false>(v);
  {
    unsigned char* d = buf + PL::rk_fw(lt, row);
#pragma unroll
    for (int k = 0; k < E; ++k) *reinterpret_cast<float2*>(d + 256 * k) = v[k];
  }
  __syncthreads();
  // the exchange also turns the CTA: lanes now run along the rows, so each frequency is stored contiguously
  const int row2 = threadIdx.x % RB3, lt2 = threadIdx.x / RB3, iq2 = blockIdx.x * RB3 + row2;
  plane_fwd8<P>(v, tw, lt2, [&](int q, int r) {
    return *reinterpret_cast<const float2*>(buf + PL::rk_fr(lt2, row2, r) + 2048 * q);
  });
  if (iq2 >= nrows) return;
  float2* dst = R + (long long)blockIdx.y * P * nrows + iq2;
#pragma unroll
  for (int q = 0; q < Q; ++q)
#pragma unroll
    for (int r = 0; r < NT; ++r) dst[(long long)(lt2 + NT * q + E * r) * nrows] = v[NT * q + r];
}

// One (transform, kx) plane of R: n x n values in and out.
template <int P, bool ADJ>
__global__ void __launch_bounds__(Plane<P>::THREADS, Plane<P>::MINB)
    conv3_plane(const int* __restrict__ active, const float2* __restrict__ tw_g, const float2* __restrict__ gplane,
                float2* __restrict__ R, int n, int tx0, int tx_div) {
  typedef Plane<P> PL;
  constexpr int E = PL::E, NT = PL::NT, Q = PL::Q, H = PL::H, PB = PL::PB, M = PL::M;
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ float2 tw[PL::TW];
  pdl_trigger();
  pdl_wait();
  const int tx = tx0 + blockIdx.y;
  if (active && !active[tx_div > 1 ? tx / tx_div : tx]) return;
  plane_twiddles<P>(tw, tw_g, PL::THREADS);
  __syncthreads();
  auto at = [&](int o) -> float2& { return *reinterpret_cast<float2*>(smem + o); };
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int STEP = PL::THREADS / NT;  // transforms in flight
  float2* base = R + ((long long)blockIdx.y * P + blockIdx.x) * n * n;
  float2 v[E];
  // y direction: rows z, z + 2 | z + 1, z + 3 in the half-warps
  const int lr = lane % NT, zr = ((lane >> 3) & 1) * 2 + (lane >> 4);
  for (int z0 = 4 * warp; z0 < n; z0 += STEP) {
    const int z = z0 + zr;
    const float2* src = base + z * n;
    const int nat = PL::row_nat(z, lr), fw = PL::row_fw(z, lr);
    const bool ok = z < n;
#pragma unroll
    for (int r = 0; r < E / 2; ++r) {
      const int y = lr + NT * r;
      v[r] = ok && y < n ? src[y] : make_float2(0.f, 0.f);
    }
    dft_n_lo<E, false>(v);
#pragma unroll
    for (int k = 0; k < E; ++k) at(fw ^ PL::row_fw_k(k)) = v[k];
    __syncwarp();
    plane_fwd8<P>(v, tw, lr, [&](int q, int r) { return at(nat ^ PL::row_fr_k(q, r)); });
    __syncwarp();
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
      for (int r = 0; r < NT; ++r) at(nat ^ PL::row_nat_k(q, r)) = v[NT * q + r];
  }
  __syncthreads();
  // z direction: columns ky = c0 + w of the warp, 8 lanes each
  const int w = lane & 3, lc = lane >> 2, xc = 4 * warp + w;
  const int kxm = blockIdx.x <= H ? blockIdx.x : P - blockIdx.x;
  const int rx = PL::col_rx(lc, xc);
  for (int c0 = 4 * warp; c0 < P; c0 += STEP) {
    const int ky = c0 + w, rs = PL::col_r(lc, ky);
#pragma unroll
    for (int r = 0; r < E / 2; ++r) v[r] = lc + NT * r < n ? at(rs + NT * r * PB) : make_float2(0.f, 0.f);
    dft_n_lo<E, false>(v);
    __syncwarp();  // the column's slots are free once all of its lanes have read them
    {
      const int fw = PL::col_fw(lc, ky, xc);
#pragma unroll
      for (int k = 0; k < E; ++k) at((fw ^ ((k & 3) * M)) + (k >> 2) * 4 * PB) = v[k];
    }
    __syncwarp();
    plane_fwd8<P>(v, tw, lc, [&](int q, int r) {
      return at(((PL::fr_up(r) ? rx : rs) ^ ((r & 3) * M)) + PL::fr_off(q, r));
    });
    // frequencies kz = lc + 8 q + E r, folded to P - kz from P / 2 on
    const float2* glo = gplane + ((long long)kxm * (P / 4) + (c0 >> 2)) * ((H + 1) * 4) + 4 * lc + w;
    const float2* ghi = glo + 4 * (P - 2 * lc);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
#pragma unroll
      for (int r = 0; r < NT; ++r) {
        const int k0 = NT * q + E * r;
        float2 g = __ldg(k0 < H ? glo + 4 * k0 : ghi - 4 * k0);
        if (ADJ) g.y = -g.y;
        v[NT * q + r] = c_mul(v[NT * q + r], g);
      }
      dft8<true, true>(v + NT * q);
    }
    __syncwarp();  // the forward exchange has been read
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int iw = PL::col_iw(lc, q, ky, xc);
#pragma unroll
      for (int s = 0; s < NT; ++s) at((iw ^ ((s & 3) * M)) + (s >> 2) * 4 * PB) = v[NT * q + s];
    }
    __syncwarp();
    plane_invE<P>(v, tw, lc, [&](int r) { return at(((PL::ir_up(r) ? rx : rs) ^ ((r & 3) * M)) + PL::ir_off(r)); });
    __syncwarp();
#pragma unroll
    for (int k = 0; k < E / 2; ++k)
      if (lc + NT * k < n) at(rs + NT * k * PB) = v[k];
    __syncwarp();
  }
  __syncthreads();
  // y direction back
  for (int z0 = 4 * warp; z0 < n; z0 += STEP) {
    const int z = z0 + zr;
    const int nat = PL::row_nat(z, lr), iw = PL::row_iw(z, lr);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
#pragma unroll
      for (int r = 0; r < NT; ++r) v[NT * q + r] = at(nat ^ PL::row_nat_k(q, r));
      dft8<true, true>(v + NT * q);
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
      for (int s = 0; s < NT; ++s) at(iw ^ PL::row_iw_k(q, s)) = v[NT * q + s];
    __syncwarp();
    plane_invE<P>(v, tw, lr, [&](int r) { return at(nat ^ PL::row_ir_k(r)); });
    if (z < n) {
      float2* dst = base + z * n;
#pragma unroll
      for (int k = 0; k < E / 2; ++k) {
        const int y = lr + NT * k;
        if (y < n) dst[y] = v[k];
      }
    }
  }
}

// ghat [kz][ky][kx] into the planes of PlaneLayout::GPLANE: plane kx, kz and ky as its other two axes
template <int P>
__global__ void plane_ghat_kernel(const float2* __restrict__ ghat, float2* __restrict__ gplane) {
  constexpr int H = P / 2;
  const int i = blockIdx.x * blockDim.x + threadIdx.x, kx = blockIdx.y;
  if (i >= Plane<P>::GPLANE) return;
  const int kz = (i >> 2) % (H + 1), ky = 4 * ((i >> 2) / (H + 1)) + (i & 3);
  gplane[(long long)kx * Plane<P>::GPLANE + i] = ghat[((long long)kz * P + ky) * P + kx];
}

template <int P, int EPI, int DK>
__global__ void __launch_bounds__(256) conv3_rows_inv(const ConvOp op, const float2* __restrict__ tw_g,
                                                      const float2* __restrict__ R, int n, int nrows, int nblk) {
  typedef Plane<P> PL;
  constexpr int E = PL::E, NT = PL::NT, Q = PL::Q;
  __shared__ float2 tw[PL::TW];
  __shared__ __align__(16) unsigned char buf[P * RB3 * 8];
  pdl_trigger();
  pdl_wait();
  const int tx = op.tx0 + blockIdx.y;
  if (op.active && !op.active[op.tx_div > 1 ? tx / op.tx_div : tx]) return;
  plane_twiddles<P>(tw, tw_g, 256);
  float2 v[E];
  {
    const int row = threadIdx.x % RB3, lt = threadIdx.x / RB3, iq = blockIdx.x * RB3 + row;
    const float2* src = R + (long long)blockIdx.y * P * nrows + iq;
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
      for (int r = 0; r < NT; ++r)
        v[NT * q + r] = iq < nrows ? src[(long long)(lt + NT * q + E * r) * nrows] : make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      dft8<true, true>(v + NT * q);
#pragma unroll
      for (int k = 0; k < NT; ++k) *reinterpret_cast<float2*>(buf + PL::rk_iw(lt, row, k) + 16384 * q) = v[NT * q + k];
    }
  }
  const int lt = threadIdx.x % NT, row = threadIdx.x / NT, iq = blockIdx.x * RB3 + row;
  const bool rowok = iq < nrows;
  const long long row0 = (long long)(rowok ? iq : 0) * n, base = (long long)tx * nrows * n + row0;
  const bool postf = op.mul_f && op.adjoint;
  bool need_aux = EPI == EPI_RESID || (EPI == EPI_CONV_ADD && op.aux) || DK == DOTS_RV || DK == DOTS_RES;
  if (DK == DOTS_ANY)
    for (int s = 0; s < DOT_SLOTS; ++s) need_aux |= op.dot_a[s] == OP_AUX || op.dot_b[s] == OP_AUX;
  // epilogue operands are loaded before the exchange so their latency overlaps it
  float2 pre_src[E / 2], pre_aux[E / 2];
#pragma unroll
  for (int k = 0; k < E / 2; ++k) {
    const int ix = lt + NT * k;
    const bool ok = rowok && ix < n;
    pre_src[k] = (ok && EPI != EPI_CONV_ADD) ? op.esrc[base + ix] : make_float2(0.f, 0.f);
    pre_aux[k] = (ok && need_aux) ? op.aux[base + ix] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  {
    const unsigned char* d = buf + PL::rk_ir(lt, row);
    plane_invE<P>(v, tw, lt, [&](int r) { return *reinterpret_cast<const float2*>(d + 2048 * r); });
  }
  float2 acc[DOT_SLOTS];
#pragma unroll
  for (int s = 0; s < DOT_SLOTS; ++s) acc[s] = make_float2(0.f, 0.f);
#pragma unroll
  for (int k = 0; k < E / 2; ++k) {
    const int ix = lt + NT * k;
    if (!rowok || ix >= n) continue;
    const long long idx = base + ix;
    float2 c = v[k];
    if (EPI == EPI_RESID && op.gz) op.gz[idx] = c_add(c, op.zadd[idx]);
    if (postf) c = c_cjmul(op.f[row0 + ix], c);
    const float2 src = pre_src[k], aux = pre_aux[k];
    float2 y;
    if (EPI == EPI_MATVEC) {
      y = c_sub(src, c);
    } else if (EPI == EPI_RESID) {
      y = c_sub(aux, c_sub(src, c));
    } else {
      y = c_add(c, aux);
    }
    op.out[idx] = y;
    if (op.out2) op.out2[idx] = y;
    dots_accumulate<DK>(op, acc, y, src, aux);
  }
  if constexpr (DK != DOTS_NONE)
    block_dots<256, DotSlots<DK>::MASK>(acc, reinterpret_cast<float2*>(op.part) + ((size_t)tx * nblk + blockIdx.x) * DOT_SLOTS);
}

template <int P>
static cisor_status conv3_pass_t(cisor_ctx* c, const ConvOp& op) {
  typedef Plane<P> PL;
  const int n = c->n, nrows = c->nrows;
  const dim3 grow((nrows + RB3 - 1) / RB3, op.ntx), gpl(P, op.ntx);
#define CISOR_ROWS_FWD(PRO) \
  CISOR_CUDA(launch_pdl(conv3_rows_fwd<P, PRO>, grow, dim3(256), 0, c->stream, op, c->tw, c->R, n, nrows))
  switch (op.prologue) {
    case PRO_COPY: CISOR_ROWS_FWD(PRO_COPY); break;
    case PRO_PUPDATE: CISOR_ROWS_FWD(PRO_PUPDATE); break;
    default: CISOR_ROWS_FWD(PRO_AXPY); break;
  }
#undef CISOR_ROWS_FWD
  CISOR_CUDA(launch_pdl(op.adjoint ? conv3_plane<P, true> : conv3_plane<P, false>, gpl, dim3(PL::THREADS), PL::BYTES,
                        c->stream, op.active, c->tw, c->gplane, c->R, n, op.tx0, op.tx_div));
  const int dk = dots_kind(op);
#define CISOR_ROWS_INV(E, D) \
  CISOR_CUDA(launch_pdl(conv3_rows_inv<P, E, D>, grow, dim3(256), 0, c->stream, op, c->tw, c->R, n, nrows, c->nblk))
  switch (op.epilogue) {
    case EPI_MATVEC:
      if (dk == DOTS_NONE) CISOR_ROWS_INV(EPI_MATVEC, DOTS_NONE);
      else if (dk == DOTS_RV) CISOR_ROWS_INV(EPI_MATVEC, DOTS_RV);
      else if (dk == DOTS_TS) CISOR_ROWS_INV(EPI_MATVEC, DOTS_TS);
      else CISOR_ROWS_INV(EPI_MATVEC, DOTS_ANY);
      break;
    case EPI_RESID:
      if (dk == DOTS_RES) CISOR_ROWS_INV(EPI_RESID, DOTS_RES);
      else CISOR_ROWS_INV(EPI_RESID, DOTS_ANY);
      break;
    default:
      if (dk == DOTS_NONE) CISOR_ROWS_INV(EPI_CONV_ADD, DOTS_NONE);
      else CISOR_ROWS_INV(EPI_CONV_ADD, DOTS_ANY);
      break;
  }
#undef CISOR_ROWS_INV
  c->launches += 3;
  return CISOR_OK;
}

template <int P>
static cisor_status conv3_init_t() {
  CISOR_CUDA(cudaFuncSetAttribute(conv3_plane<P, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, Plane<P>::BYTES));
  CISOR_CUDA(cudaFuncSetAttribute(conv3_plane<P, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, Plane<P>::BYTES));
  return CISOR_OK;
}

template <int P>
static cisor_status conv3_tables_t(cisor_ctx* c) {
  plane_ghat_kernel<P><<<dim3((Plane<P>::GPLANE + 255) / 256, P / 2 + 1), 256, 0, c->stream>>>(c->ghat, c->gplane);
  CISOR_CUDA(cudaGetLastError());
  return CISOR_OK;
}

size_t conv3_ghat_elems(int P) { return (size_t)(P / 2 + 1) * (P == 64 ? Plane<64>::GPLANE : Plane<128>::GPLANE); }
cisor_status conv3_tables(cisor_ctx* c) { return c->P == 64 ? conv3_tables_t<64>(c) : conv3_tables_t<128>(c); }
bool conv3_ok(int dim, int P) { return dim == 3 && P <= 128; }
int conv3_rows_per_block() { return RB3; }
cisor_status conv3_init(int P) { return P == 64 ? conv3_init_t<64>() : conv3_init_t<128>(); }
cisor_status conv3_pass(cisor_ctx* c, const ConvOp& op) {
  return c->P == 64 ? conv3_pass_t<64>(c, op) : conv3_pass_t<128>(c, op);
}

}  // namespace cisor
