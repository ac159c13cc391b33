// Shared-memory layout of the 3D plane convolution (conv3d.cu) as byte
// offsets, host-visible so that its bank conflicts and its exchanges can be
// enumerated without a GPU.
//
// The plane S has P / 2 rows (z) of P values (ky); value ky of row z sits at
// slot ky ^ 4 (z & 3) of its row, so that eight lanes along a row (in two rows
// z, z + 2) as well as four rows times four columns meet 16 different banks.
// Behind it, xs holds the upper half of every column exchange for the
// THREADS / 8 columns in flight; its P / 2 rows are folded in two so that its row
// stride is S's.  Offsets are "lane part ^ constant" (rows) or "(lane part ^
// constant) + constant" (columns), so an access costs at most one integer
// instruction.  E = P / 8 elements a thread, 8 threads (lt) a transform.
#pragma once

namespace cisor {

#ifdef __CUDACC__
#define CISOR_HD static __host__ __device__ __forceinline__ constexpr
#else
#define CISOR_HD static inline constexpr
#endif

template <int P> struct PlaneLayout {
  static constexpr int E = P / 8, NT = 8, Q = E / NT, H = P / 2;
  static constexpr int PB = 8 * P;      // bytes of a row
  static constexpr int XOFF = H * PB;   // xs
  static constexpr int XCOLS = P / 2;   // columns in flight
  static constexpr int THREADS = XCOLS * NT;
  static constexpr int BYTES = XOFF + H * XCOLS * 8;
  static constexpr int M = PB + 32;     // exchange rows are permuted by their two low bits, columns by 4 times them

  // ---- row transforms of plane row z
  CISOR_HD int zz(int z) { return 4 * (z & 3); }
  // natural order: value lt + 8 q + E r
  CISOR_HD int row_nat(int z, int lt) { return z * PB + 8 * (lt ^ zz(z)); }
  CISOR_HD int row_nat_k(int q, int r) { return 8 * (NT * q + E * r); }
  // forward exchange: value E lt + k written, j + E r read (j = lt + 8 q)
  CISOR_HD int row_fw(int z, int lt) { return z * PB + 8 * ((E * lt + lt) ^ zz(z)); }
  CISOR_HD int row_fw_k(int k) { return 8 * k; }
  CISOR_HD int row_fr_k(int q, int r) { return 8 * ((E * r + r) ^ (NT * q)); }  // from row_nat
  // inverse exchange: value 8 j + s written, lt + 8 r read
  CISOR_HD int row_iw(int z, int lt) { return z * PB + 8 * ((NT * lt + lt) ^ zz(z)); }
  CISOR_HD int row_iw_k(int q, int s) { return 8 * (NT * NT * q + s); }
  CISOR_HD int row_ir_k(int r) { return 8 * (NT * r + (r & 7)); }  // from row_nat

  // ---- column transforms: plane column c, column xc of xs
  CISOR_HD int xrow(int row) { return (row % (H / 2)) * PB + (row / (H / 2)) * (PB / 2); }
  CISOR_HD int part(int row, int c, int l3) { return row * PB + 8 * (c ^ (4 * l3)); }
  CISOR_HD int xpart(int row, int xc, int l3) { return XOFF + xrow(row) + 8 * (xc ^ (4 * l3)); }
  // lane bases of reads (and of natural order: value lt + 8 r at + 8 r PB)
  CISOR_HD int col_r(int lt, int c) { return part(lt, c, lt & 3); }
  CISOR_HD int col_rx(int lt, int xc) { return xpart(lt, xc, lt & 3); }
  // forward exchange: value E lt + k at (base ^ k3 M) + (k >> 2) 4 PB; value j + E r at (base ^ r3 M) + offset
  CISOR_HD int col_fw(int lt, int c, int xc) {
    return lt < NT / 2 ? part(E * lt + (lt & 3), c, lt & 3) : xpart(E * (lt - NT / 2) + (lt & 3), xc, lt & 3);
  }
  CISOR_HD bool fr_up(int r) { return r >= NT / 2; }
  CISOR_HD int fr_off(int q, int r) { return fr_up(r) ? xrow(E * (r - NT / 2) + NT * q) : (E * r + NT * q) * PB; }
  // inverse exchange: value 8 j + s likewise from the base of group q; value lt + 8 r from the read bases
  CISOR_HD int col_iw(int lt, int q, int c, int xc) {
    return E == 16 ? (q == 0 ? part(NT * lt + (lt & 3), c, lt & 3) : xpart(NT * lt + (lt & 3), xc, lt & 3))
                   : (lt < NT / 2 ? part(NT * lt + (lt & 3), c, lt & 3) : xpart(NT * (lt - NT / 2) + (lt & 3), xc, lt & 3));
  }
  CISOR_HD bool ir_up(int r) { return r >= E / 2; }
  CISOR_HD int ir_off(int r) { return ir_up(r) ? xrow(NT * (r - E / 2)) : NT * r * PB; }

  // ---- exchange of the row kernels, [P][32] values: row transforms of 32 rows, lanes along lt on one side and
  // along the rows on the other
  CISOR_HD int rk_fw(int lt, int row) { return 8 * (32 * E * lt + (row ^ (2 * lt))); }  // value E lt + k: + 256 k
  CISOR_HD int rk_fr(int lt, int row, int r) { return 8 * (32 * (lt + E * r) + (row ^ (2 * r))); }  // + 2048 q
  CISOR_HD int rk_iw(int lt, int row, int s) { return 8 * (32 * (NT * lt + s) + (row ^ (2 * s))); }  // + 16384 q
  CISOR_HD int rk_ir(int lt, int row) { return 8 * (32 * lt + (row ^ (2 * lt))); }  // value lt + 8 r: + 2048 r

  // ---- stage twiddles w^(r j), r < 8, j < E, in rows of E + 1
  CISOR_HD int tw(int r, int j) { return r * (E + 1) + j; }
  static constexpr int TW = NT * (E + 1);

  // ---- ghat planes [kx <= H][ky / 4][kz <= H][ky % 4]: 8 lanes along kz and 4 along ky read 256 contiguous bytes
  static constexpr int GPLANE = (P / 4) * (H + 1) * 4;
};

}  // namespace cisor
