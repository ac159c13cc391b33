// The sensing GEMMs (Eq. 5 forward, Eq. 13's H^H w adjoint) on the fifth-
// generation tensor cores, TF32 with a hi / lo split: every FP32 operand x is
// held as hi = x with its 13 low mantissa bits cleared (exactly a TF32 value)
// and lo = x - hi (exact in FP32, read as TF32 by the MMA), and a product is
// hi.hi + lo.hi + hi.lo: about 21 mantissa bits; with the accumulation below
// the GEMMs are within 8e-7 of an FP64 product, inside the 1e-5 sensing
// tolerance that a single TF32 or a BF16 hi / lo product (1.5e-5) misses.
//
// The complex GEMM is one real GEMM: H is read as interleaved (Re, Im) floats,
// K = 2 x (complex columns), and each transmitter t contributes two rows of the
// small operand, so that D[row][2t] and D[row][2t + 1] are Re and Im of its
// result:
//   forward  Y[t][m] = sum_n H[m][n] X_t[n], X_t = f u_t (Eq. 5):
//            rows 2t = (Re X, -Im X), 2t + 1 = (Im X, Re X) per n
//   adjoint  z_t[n] = sum_m conj(H[m][n]) w_t[m] (H^H w, Eq. 13), read from the
//            transposed copy Ht[n][m] so that both GEMMs stream K-major rows:
//            rows 2t = (Re w, Im w), 2t + 1 = (Im w, -Re w) per m
// An accumulator tile is 128 rows of the big operand (receivers forward, field
// entries adjoint) by 2T columns (rounded up to NB) in tensor memory, and K is
// streamed in chunks of 32 floats.  The forward pass splits K into slabs
// (partials [split][T][M] summed by sense_reduce_kernel, in a fixed order); an
// adjoint tile covers all of K (2M) and writes z and conj(f) z.
//
// Up to 96 transmitters (NB <= 192) H and Ht are stored as those tiles: 128 rows
// by 32 floats, contiguous, in the order in which a CTA streams them (tile_off), so
// that a chunk is one 16 KB bulk copy by one thread (sense_tile.cuh); the copies
// alone, which only read, run at 7.3 TB/s (a copy that also writes moves 6.8).  One
// warp-specialised CTA per SM runs over the tiles (sense_ws_kernel): a thread keeps SENSE_STAGES bulk copies of the big operand in flight, converter
// warps split each chunk into hi / lo planes in TENSOR MEMORY, builder warps write
// the small operand's planes to shared memory, two threads issue the MMAs (A from
// tensor memory, B from shared memory) and the remaining warps add finished chunks
// into FP32 registers; several buffers of everything behind the load ring let all
// roles work on different chunks at once.  A in tensor memory is what makes the
// shared-memory pipe suffice: per 16 KB chunk it carries the copy, one read, the
// small operand's write and its reads by the MMAs (93 KB at NB = 96 against 140 KB
// with both planes of A there).
// Measured at 48 transmitters, 1024 receivers, 64^3 (H and Ht of 2.1 GB): forward
// 1.15 -> 0.60 ms, adjoint 0.93 -> 0.58 ms against the kernel below on row-major
// matrices, which does all roles in every thread; 64 transmitters, 256 receivers,
// 256^2: 0.136 -> 0.071, 0.092 -> 0.082; 81, 36, 32^3 vectorial: 0.108 -> 0.095,
// 0.096 -> 0.065; 8, 360, 128^2: 0.044 -> 0.022, 0.037 -> 0.017; 8, 32, 64^2: 0.017 -> 0.014,
// 0.008 -> 0.007 (all launches; slower only with a few receivers and many
// transmitters, whose chunk is computed whole however narrow it is: 48, 2, 256^2
// adjoint 20 -> 23 us).  What bounds it: the hand-overs between the roles (below); the MMAs keep
// the tensor pipe about half of the time at NB = 96, the copies the memory for
// half.  More than 96 transmitters leave no room for two
// accumulators and A in tensor memory and take the kernel below (sense_tc_kernel).
// Every wait is bounded (a timeout sets the context's error flag, read by the host
// after the call).
#include "common.cuh"
#include "sense_tile.cuh"
#include "tc5.cuh"

namespace cisor {

constexpr int SLBO = 144, SSBO = 8 * SLBO;   // K-group and 8-row strides of the operand tiles (bytes)
constexpr int SPA = 16 * SSBO;               // bytes of one plane of the 128-row tile
constexpr int STH = 256;                     // threads per CTA
constexpr int S_WAIT = 1 << 20;              // polls of the MMA completion barrier before giving up
// K (floats) per split of the forward GEMM, at most.  sense_tc_kernel, a CTA per split and row tile: splits of 64 chunks,
// 2048 and more CTAs at 48 transmitters, 1024 receivers, 64^3, measured faster than one wave of 432-chunk CTAs (1.04
// against 1.59 ms): CTAs that start together read the same slab of the small operand, which then stays in L2 while H
// streams past it.  sense_ws_kernel, whose persistent CTAs take splits as items, in the same order: 16, 32 and 64 chunks
// 594 us there, 128 564, 256 628; 64, 256, 256^2 87, 78, 67, 67, 67.
constexpr long long S_KMAX = 64 * SK;
constexpr long long S_MAX = 256;  // at most this many splits (partials T x M x 8 bytes each)


__host__ __device__ constexpr int soff(int row, int k) {
  return (row >> 3) * SSBO + (k >> 2) * SLBO + (row & 7) * 16 + (k & 3) * 4;
}
__device__ __forceinline__ float tf32_hi(float x) { return __uint_as_float(__float_as_uint(x) & 0xFFFFE000u); }
__device__ __forceinline__ long long wrap(long long j, long long NP) {
  while (j >= NP) j -= NP;
  return j;
}

// accumulator columns for ntx transmitters (2 ntx rounded up to an instantiated width)
int sense_tc_cols(int ntx) {
  const int need = 2 * ntx;
  return need <= 32 ? 32 : need <= 64 ? 64 : need <= 96 ? 96 : need <= 128 ? 128 : need <= 192 ? 192 : 256;
}
constexpr int WS_NB = 192;  // most accumulator columns of the warp-specialised kernel: 2 x 192 and A's 128 fill the 512

// ADJ = 0: A = H [rows = M][lda = 2 Nf], K range [ks KS, ks KS + KS) of 2 Nf, small operand from f and u [T][Nf];
//          out0 = partials [(ks T + t) M + m].
// ADJ = 1: A = Ht [rows = Nf][lda = 2 M], all of K = 2 M, small operand from w [T][M];
//          out0 = z [t Nf + n], out1 (may be null) = conj(f) z.
// For more than 96 and up to 128 transmitters: NB = 256 accumulator columns.  Each chunk's 12 MMAs start a
// fresh accumulator, alternating between two TMEM buffers: while chunk c's MMAs run, the threads add chunk
// c - 1's result into FP32 registers (round to nearest).  The tensor cores' FP32 accumulation rounds its sums
// more coarsely: accumulating a whole split in TMEM (64 to 432 chunks, hundreds of MMAs) left the products
// 1.2e-5 to 1.5e-5 from FP64 on random inputs; with chains of 12 they are within 8e-7 (C2, C3 sizes).
constexpr int TC_NB = 256, TC_SMEM = 2 * SPA + 2 * (TC_NB / 8) * SSBO;
template <int ADJ>
__global__ void __launch_bounds__(STH, 1) sense_tc_kernel(const float* __restrict__ A, long long lda, long long rows,
                                                       long long K, long long KS, const float2* __restrict__ src,
                                                       long long lds, const float2* __restrict__ f, long long NP,
                                                       int T, int M, long long Nf, float2* __restrict__ out0,
                                                       float2* __restrict__ out1, int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tslot;
  constexpr int NB = TC_NB, SPB = (NB / 8) * SSBO;
  constexpr int NH = NB / 2;  // accumulator columns per thread
  constexpr uint32_t ncol = 2 * NB;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long row0 = (long long)blockIdx.x * 128;
  const long long kb = ADJ ? 0 : (long long)blockIdx.y * KS;
  const long long ke = ADJ ? K : (kb + KS < K ? kb + KS : K);
  const int nch = (int)((ke - kb + SK - 1) / SK);
  unsigned char* sb = sm + 2 * SPA;
  for (int i = tid * 16; i < 2 * SPB; i += STH * 16) *reinterpret_cast<uint4*>(sb + i) = make_uint4(0, 0, 0, 0);
  if (tid == 0) mbar_init(&mbar);
  if (warp == 0) tmem_alloc(&tslot, ncol);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tslot, s0 = smem_addr(sm);
  const int nitems = T * 16;  // (transmitter, complex column) pairs of a chunk
  float4 ra[4];
  float2 rb[8], rf[8];
  auto fetch = [&](long long k0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int idx = tid + STH * q, r = idx >> 3, kg = idx & 7;
      const long long gr = row0 + r, kk = k0 + 4 * kg;
      ra[q] = (gr < rows && kk < ke) ? __ldg(reinterpret_cast<const float4*>(A + gr * lda + kk))
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int item = tid + STH * q;
      const long long j = k0 / 2 + (item & 15);
      const bool ok = item < nitems && 2 * j < ke;
      rb[q] = ok ? __ldg(src + (long long)(item >> 4) * lds + j) : make_float2(0.f, 0.f);
      if (!ADJ) rf[q] = ok ? __ldg(f + wrap(j, NP)) : make_float2(0.f, 0.f);
    }
  };
  auto stage = [&]() {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int idx = tid + STH * q, o = soff(idx >> 3, 4 * (idx & 7));
      const float4 x = ra[q];
      const float4 h = make_float4(tf32_hi(x.x), tf32_hi(x.y), tf32_hi(x.z), tf32_hi(x.w));
      *reinterpret_cast<float4*>(sm + o) = h;
      *reinterpret_cast<float4*>(sm + SPA + o) = make_float4(x.x - h.x, x.y - h.y, x.z - h.z, x.w - h.w);
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int item = tid + STH * q;
      if (item < nitems) {
        const int c = item & 15, t = item >> 4;
        const float2 x = ADJ ? rb[q] : c_mul(rf[q], rb[q]);
        const float2 e0 = ADJ ? x : make_float2(x.x, -x.y);
        const float2 e1 = ADJ ? make_float2(x.y, -x.x) : make_float2(x.y, x.x);
        const int o0 = soff(2 * t, 2 * c), o1 = soff(2 * t + 1, 2 * c);
        const float2 h0 = make_float2(tf32_hi(e0.x), tf32_hi(e0.y)), h1 = make_float2(tf32_hi(e1.x), tf32_hi(e1.y));
        *reinterpret_cast<float2*>(sb + o0) = h0;
        *reinterpret_cast<float2*>(sb + SPB + o0) = make_float2(e0.x - h0.x, e0.y - h0.y);
        *reinterpret_cast<float2*>(sb + o1) = h1;
        *reinterpret_cast<float2*>(sb + SPB + o1) = make_float2(e1.x - h1.x, e1.y - h1.y);
      }
    }
  };
  uint32_t ph = 0;
  bool failed = false;
  auto wait_mma = [&]() {
    const bool ok = mbar_wait(&mbar, ph, S_WAIT);
    ph ^= 1u;
    tc_fence_after();
    if (__syncthreads_or(!ok)) {
      if (tid == 0) *reinterpret_cast<volatile int*>(err) = 1;  // mapped host memory: a plain store
      failed = true;
    }
    return !failed;
  };
  const uint32_t id = tc_idesc_tf32(128, NB);
  // row 32 (w % 4) + lane of the tile in this warp's TMEM lane quarter; warps w, w + 4 split the columns
  const int q = warp & 3, half = warp >> 2;
  const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16) + half * NH;
  float acc[NH];
#pragma unroll
  for (int j = 0; j < NH; ++j) acc[j] = 0.f;
  auto gather = [&](int buf) {  // acc += this thread's columns of accumulator buffer buf
#pragma unroll
    for (int c0 = 0; c0 < NH; c0 += 8) {
      float d[8];
      tmem_ld8(tl + buf * NB + c0, d);
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[c0 + j] += d[j];
    }
  };
  fetch(kb);
  for (int ch = 0; ch < nch; ++ch) {
    if (ch > 0 && !wait_mma()) break;  // the previous chunk's MMAs have read the tiles
    stage();
    if (ch + 1 < nch) fetch(kb + (long long)(ch + 1) * SK);
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0) {
      const uint32_t d = tmem + (ch & 1) * NB;
#pragma unroll
      for (int ks = 0; ks < SK / 8; ++ks) {
        const uint32_t ah = s0 + ks * 2 * SLBO, al = ah + SPA;
        const uint32_t bh = s0 + 2 * SPA + ks * 2 * SLBO, bl = bh + SPB;
        const uint64_t dah = tc_desc(ah, SLBO, SSBO), dbh = tc_desc(bh, SLBO, SSBO);
        tc_mma_tf32(d, dah, dbh, id, ks > 0 ? 1u : 0u);
        tc_mma_tf32(d, tc_desc(al, SLBO, SSBO), dbh, id, 1u);
        tc_mma_tf32(d, dah, tc_desc(bl, SLBO, SSBO), id, 1u);
      }
      tc_commit(&mbar);
    }
    if (ch > 0) gather((ch - 1) & 1);  // the previous chunk's result, while this chunk's MMAs run
  }
  if (!failed && nch > 0 && wait_mma()) gather((nch - 1) & 1);
  if (!failed) {
    const long long row = row0 + 32 * q + lane;
#pragma unroll
    for (int c0 = 0; c0 < NH; c0 += 2) {
      {
        const int t = (half * NH + c0) / 2;
        if (t < T && row < rows) {
          const float2 v = make_float2(acc[c0], acc[c0 + 1]);
          if (!ADJ) {
            out0[((long long)blockIdx.y * T + t) * M + row] = v;
          } else {
            out0[(long long)t * Nf + row] = v;
            if (out1) out1[(long long)t * Nf + row] = c_cjmul(__ldg(f + wrap(row, NP)), v);
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, ncol);
}

// ------------------------------------------------------------------ warp-specialised kernel, NB <= 192
// Up to 128 columns: warps 0-7 are A converters, two groups of four on alternate chunks (thread = tile row =
// tensor-memory lane), 8-15 accumulate (lane quarter w % 4, columns halved), 16-23 build B, two groups on alternate
// chunks.  192 columns: 4 converters, 12 accumulators (thirds of the columns: 96 a thread would spill), 4 builders.
// Then the producer of the bulk copies and two MMA issuers.
// Chunk n of the CTA's sequence over all its tiles uses load stage n % SENSE_STAGES, operand buffer n % DEP (A in
// tensor memory, B in shared memory) and accumulator n % ND.  An MMA issuer waits once a chunk: `ready` collects the
// converters', the builders' and the accumulators' arrivals (the last for the chunk ND before, whose accumulator this
// one reuses).  A completed barrier still costs its waiter 200 to 350 cycles and a commit 300, against about 650 for
// the chunk's MMAs at NB = 96; that is why the roles run up to DEP chunks apart and why two threads issue, each
// waiting while the other's MMAs run.  Forward / adjoint at 48 transmitters, 64^3: 0.99 / 0.80 ms with one group of
// builders and one issuer, 0.73 / 0.64 with two groups, 0.67 / 0.58 with two issuers
// (all before the reduction's faster sums, with which it is 0.60 / 0.58).
// operand buffers and accumulators (at most as many): what 512 columns of tensor memory hold.  An even number of
// buffers: then a buffer's chunks belong to one group of converters and of builders and to one issuer, so that nobody
// tests a barrier that is still a phase behind the one it waits for.
__host__ __device__ constexpr int ws_dep(int nb) { return nb <= 96 ? 4 : 2; }
__host__ __device__ constexpr int ws_nd(int nb) { return nb <= 64 ? 4 : 2; }
__host__ __device__ constexpr int ws_groups(int nb) { return nb <= 128 ? 2 : 1; }  // of four builder warps, and of four converters
constexpr int WS_ISS = 2;  // MMA issuers, on alternate chunks
__host__ __device__ constexpr int ws_threads(int nb) { return (17 + WS_ISS + 4 * ws_groups(nb)) * 32; }
constexpr int SENSE_STAGES = 6;
constexpr int WS_A = 128 * SK * 4;  // bytes of a chunk of A
constexpr int ws_smem(int nb) { return 1024 + SENSE_STAGES * WS_A + ws_dep(nb) * 2 * (nb / 8) * SSBO; }

struct WsBars {
  uint64_t full[SENSE_STAGES], empty[SENSE_STAGES], ready[4], done[4];
  int pieces[SENSE_STAGES];  // 16-byte pieces a row of the chunk in each load stage, where rows end in a narrow chunk
};

// NARROW: rows end in a chunk narrower than SK (tile_kp).  Compiled apart, since finding the chunk's width costs the
// converters of every chunk: forward products of 64 transmitters, 256^2 36 -> 39 us with it, of one 23.4 -> 24.6.
template <int ADJ, int NB, bool NARROW>
__global__ void __launch_bounds__(ws_threads(NB), 1) sense_ws_kernel(const float* __restrict__ A, long long rows, int rtiles,
                                                            int nitems, long long K, long long KS,
                                                            const float2* __restrict__ src, long long lds,
                                                            const float2* __restrict__ f, long long NP, int T, int M,
                                                            long long Nf, float2* __restrict__ out0,
                                                            float2* __restrict__ out1, int* __restrict__ err) {
  extern __shared__ unsigned char smraw[];
  __shared__ __align__(8) WsBars bar;
  __shared__ uint32_t tslot;
  __shared__ volatile int failed;
  unsigned char* sm = smraw + ((1024 - (smem_addr(smraw) & 1023)) & 1023);
  constexpr int SPB = (NB / 8) * SSBO;   // bytes of a plane of B
  constexpr int IPT = NB / 32;           // (transmitter, two complex columns) pieces per building thread
  constexpr int DEP = ws_dep(NB), ND = ws_nd(NB), GB = ws_groups(NB), TH = ws_threads(NB);
  constexpr int NH = NB / (4 - GB);      // accumulator columns per accumulating thread
  constexpr uint32_t ACOL = ND * NB;     // tensor memory: ND accumulators, then DEP x (hi, lo) of A
  static_assert(ND * NB + 64 * DEP <= 512 && ND <= DEP, "tensor memory columns");
  static_assert(DEP % 2 == 0 && SENSE_STAGES % 2 == 0, "a buffer or stage belongs to one group, one issuer");
  unsigned char* sb = sm + SENSE_STAGES * WS_A;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid * 16; i < 2 * DEP * SPB; i += TH * 16) *reinterpret_cast<uint4*>(sb + i) = make_uint4(0, 0, 0, 0);
  if (tid == 0) {
    failed = 0;
    for (int i = 0; i < SENSE_STAGES; ++i) {
      mbar_init(&bar.full[i]);
      mbar_init(&bar.empty[i], 4);
    }
    for (int i = 0; i < DEP; ++i) {
      mbar_init(&bar.ready[i], 4 + 4 + 4 * (4 - GB));
      mbar_init(&bar.done[i]);
    }
  }
  if (warp == 0) tmem_alloc(&tslot, 512);
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tslot;
  // false (and everyone told) if a wait gave up, here or in another role
  auto wait = [&](uint64_t* b, uint32_t use) {
    for (int it = 0; it < S_WAIT; ++it) {
      if (mbar_wait(b, use & 1, 1)) return true;
      if (failed) return false;
    }
    failed = 1;
    *reinterpret_cast<volatile int*>(err) = 1;  // mapped host memory: a plain store
    return false;
  };
  auto wait_warp = [&](uint64_t* b, uint32_t use) { return (bool)__all_sync(0xffffffffu, wait(b, use)); };
  auto arrive = [&](uint64_t* b) {  // one arrival per warp, after all of its lanes
    __syncwarp();
    if (lane == 0) mbar_arrive(b);
  };
  // this CTA's tiles: row tile, first and last K of the slab, chunks
  struct Item {
    long long row0, kb, ke;
    int split, nch;
  };
  auto item = [&](int it) {
    Item r;
    r.split = ADJ ? 0 : it / rtiles;
    r.row0 = (long long)(ADJ ? it : it % rtiles) * 128;
    r.kb = r.split * KS;
    r.ke = r.kb + KS < K ? r.kb + KS : K;
    r.nch = (int)((r.ke - r.kb + SK - 1) / SK);
    return r;
  };
  uint32_t total = 0;  // chunks of this CTA
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) total += item(it).nch;
  if (warp < 4 * GB) {  // ---- converters: hi / lo planes of a chunk of A into tensor memory
    const int row = 32 * (warp & 3) + lane;
    const uint32_t ta = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + ACOL;
    for (uint32_t n = warp >> 2; n < total; n += GB) {
      const uint32_t s = n % SENSE_STAGES, buf = n % DEP, k = n / DEP;
      if (!wait_warp(&bar.full[s], n / SENSE_STAGES)) break;
      const int pieces = NARROW ? *(volatile int*)&bar.pieces[s] : SK / 4, z = tile_swz(row, pieces);
      const unsigned char* p = sm + s * WS_A + row * pieces * 16;  // (tile_piece)
      uint32_t h[32], l[32];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);  // behind the row's end, where B's zeros would not cancel an infinity
        if (j < pieces) x = *reinterpret_cast<const float4*>(p + ((j ^ z) << 4));
        const float v[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float hi = tf32_hi(v[e]);
          h[4 * j + e] = __float_as_uint(hi);
          l[4 * j + e] = __float_as_uint(v[e] - hi);
        }
      }
      if (k >= 1 && !wait_warp(&bar.done[buf], k - 1)) break;  // the planes' last reader
      tc_fence_after();
      tmem_st32(ta + 64 * buf, h);
      tmem_st32(ta + 64 * buf + 32, l);
      arrive(&bar.empty[s]);  // here, where the stores needed all values, not behind the loads' issue: the next copy into
                              // the stage overtook loads still on their way (wrong values in 40% of some runs)
      tmem_wait_st();
      tc_fence_before();
      arrive(&bar.ready[buf]);
    }
  } else if (warp < 16) {  // ---- accumulation
    const int q = warp & 3, part = (warp - 4 * GB) >> 2;
    const uint32_t td = tmem + ((uint32_t)(32 * q) << 16) + part * NH;
    for (int i = 0; i < ND; ++i) arrive(&bar.ready[i]);  // the first chunks' accumulators are free
    uint32_t n = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
      const Item r = item(it);
      float acc[NH];
#pragma unroll
      for (int j = 0; j < NH; ++j) acc[j] = 0.f;
      for (int ch = 0; ch < r.nch; ++ch, ++n) {
        if (!(ok = wait_warp(&bar.done[n % DEP], n / DEP))) break;
        tc_fence_after();
#pragma unroll
        for (int c0 = 0; c0 < NH; c0 += 8) {
          float d[8];
          tmem_ld8(td + n % ND * NB + c0, d);
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[c0 + j] += d[j];
        }
        tc_fence_before();
        arrive(&bar.ready[(n + ND) % DEP]);
      }
      const long long row = r.row0 + 32 * q + lane;
      if (!ok || row >= rows) continue;
#pragma unroll
      for (int c0 = 0; c0 < NH; c0 += 2) {
        const int t = (part * NH + c0) / 2;
        if (t >= T) break;
        const float2 v = make_float2(acc[c0], acc[c0 + 1]);
        if (!ADJ) {
          out0[((long long)r.split * T + t) * M + row] = v;
        } else {
          out0[(long long)t * Nf + row] = v;
          if (out1) out1[(long long)t * Nf + row] = c_cjmul(__ldg(f + wrap(row, NP)), v);
        }
      }
    }
  } else if (warp < 16 + 4 * GB) {  // ---- builders: hi / lo planes of the small operand into shared memory
    // the values of a group's next two chunks are on their way from global memory while a third is staged; a thread has
    // the columns 2 c2, 2 c2 + 1 (16 bytes; src, f and their rows are 16-byte aligned) of transmitters t0 + 16 i
    const int bt = (tid - 16 * 32) & 127, group = (warp - 16) >> 2, c2 = bt & 7, t0 = bt >> 3;
    float4 rb[2][IPT], rf[2];
    const long long step = 16 * lds;
    // the group's next chunk to fetch: tile, chunk in it, where its values lie and K left from this thread's columns on
    int fit = blockIdx.x, fch = 0, fn = 0, left = 0;
    const float2 *fp = nullptr, *ff = nullptr;
    auto enter = [&]() {
      const Item r = item(fit);
      fn = r.nch;
      left = (int)(r.ke - r.kb) - 4 * c2;
      fp = src + (long long)t0 * lds + r.kb / 2 + 2 * c2;
      if (!ADJ) ff = f + wrap(r.kb / 2 + 2 * c2, NP);
    };
    auto advance = [&](int by) {  // by chunks, over tile ends
      fch += by;
      left -= by * SK;
      fp += by * (SK / 2);
      if (!ADJ) {
        ff += by * (SK / 2);
        while (ff >= f + NP) ff -= NP;
      }
      while (fit < nitems && fch >= fn) {
        fch -= fn;
        fit += gridDim.x;
        if (fit >= nitems) break;
        enter();
        if (fch) {
          left -= fch * SK;
          fp += fch * (SK / 2);
          if (!ADJ) {
            ff += fch * (SK / 2);
            while (ff >= f + NP) ff -= NP;
          }
        }
      }
    };
    uint32_t n = group;
    auto fetch = [&](float4 (&x)[IPT], float4& fx) {
      if (fit >= nitems) return;
      const bool in = left > 0;
#pragma unroll
      for (int i = 0; i < IPT; ++i)
        x[i] = in && t0 + 16 * i < T ? __ldg(reinterpret_cast<const float4*>(fp + i * step)) : make_float4(0.f, 0.f, 0.f, 0.f);
      if (!ADJ) fx = in ? __ldg(reinterpret_cast<const float4*>(ff)) : make_float4(0.f, 0.f, 0.f, 0.f);
      advance(GB);
    };
    // stages chunk n from x, then refills x for the group's chunk after the next; false once a wait gave up
    auto build = [&](float4 (&x)[IPT], float4& fx) {
      const uint32_t buf = n % DEP, k = n / DEP;
      if (k >= 1 && !wait_warp(&bar.done[buf], k - 1)) return false;
      unsigned char* d = sb + buf * 2 * SPB;
#pragma unroll
      for (int i = 0; i < IPT; ++i) {
        const int t = t0 + 16 * i;
        if (t < T) {
          float2 v = make_float2(x[i].x, x[i].y), u = make_float2(x[i].z, x[i].w);
          if (!ADJ) {
            v = c_mul(make_float2(fx.x, fx.y), v);
            u = c_mul(make_float2(fx.z, fx.w), u);
          }
          const float hx = tf32_hi(v.x), hy = tf32_hi(v.y), gx = tf32_hi(u.x), gy = tf32_hi(u.y);
          const float lx = v.x - hx, ly = v.y - hy, kx = u.x - gx, ky = u.y - gy;
          const int o0 = soff(2 * t, 4 * c2), o1 = soff(2 * t + 1, 4 * c2);
          *reinterpret_cast<float4*>(d + o0) = ADJ ? make_float4(hx, hy, gx, gy) : make_float4(hx, -hy, gx, -gy);
          *reinterpret_cast<float4*>(d + SPB + o0) = ADJ ? make_float4(lx, ly, kx, ky) : make_float4(lx, -ly, kx, -ky);
          *reinterpret_cast<float4*>(d + o1) = ADJ ? make_float4(hy, -hx, gy, -gx) : make_float4(hy, hx, gy, gx);
          *reinterpret_cast<float4*>(d + SPB + o1) = ADJ ? make_float4(ly, -lx, ky, -kx) : make_float4(ly, lx, ky, kx);
        }
      }
      fence_async_smem();
      arrive(&bar.ready[buf]);
      fetch(x, fx);
      n += GB;
      return true;
    };
    enter();
    if (group) advance(group);
    fetch(rb[0], rf[0]);
    fetch(rb[1], rf[1]);
    while (n < total) {
      if (!build(rb[0], rf[0])) break;
      if (n < total && !build(rb[1], rf[1])) break;
    }
  } else if (warp == 16 + 4 * GB) {  // ---- producer
    if (lane == 0) {
      const long long kp = tile_kp(K);
      uint32_t n = 0;
      bool ok = true;
      for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
        const Item r = item(it);
        const int R = tile_rows(r.row0, rows);  // (rows past the last keep old values)
        const float* p = A + tile_chunk(r.row0, r.kb / SK, rows, kp);
        for (int ch = 0; ch < r.nch; ++ch, ++n, p += R * SK) {
          const uint32_t s = n % SENSE_STAGES;
          if (n >= SENSE_STAGES && !(ok = wait(&bar.empty[s], n / SENSE_STAGES - 1))) break;
          const int w = NARROW ? tile_width(r.ke - r.kb - (long long)ch * SK) : SK;
          if (NARROW) *(volatile int*)&bar.pieces[s] = w >> 2;
          mbar_expect(&bar.full[s], R * w * 4);
          bulk_load(sm + s * WS_A, p, R * w * 4, &bar.full[s]);
        }
      }
      // the loads still in flight land before the CTA's shared memory goes
      for (uint32_t m = n > SENSE_STAGES ? n - SENSE_STAGES : 0; m < n; ++m)
        (void)mbar_wait(&bar.full[m % SENSE_STAGES], (m / SENSE_STAGES) & 1, S_WAIT);
    }
    __syncwarp();
  } else {  // ---- MMA issuer
    if (lane == 0) {
      const uint32_t id = tc_idesc_tf32(128, NB), b0 = smem_addr(sb);
      uint32_t n = warp - (17 + 4 * GB);
      for (; n < total; n += WS_ISS) {
        const uint32_t buf = n % DEP;
        if (!wait(&bar.ready[buf], n / DEP)) break;
        tc_fence_after();
        const uint32_t d = tmem + n % ND * NB, a = tmem + ACOL + 64 * buf, b = b0 + buf * 2 * SPB;
#pragma unroll
        for (int ks = 0; ks < SK / 8; ++ks) {
          const uint64_t bh = tc_desc(b + ks * 2 * SLBO, SLBO, SSBO), bl = tc_desc(b + SPB + ks * 2 * SLBO, SLBO, SSBO);
          tc_mma_tf32_ts(d, a + 8 * ks, bh, id, ks > 0 ? 1u : 0u);
          tc_mma_tf32_ts(d, a + 32 + 8 * ks, bh, id, 1u);
          tc_mma_tf32_ts(d, a + 8 * ks, bl, id, 1u);
        }
        tc_commit(&bar.done[buf]);
      }
      // the MMAs still in flight end before the CTA's tensor memory goes
      if (n >= WS_ISS) (void)mbar_wait(&bar.done[(n - WS_ISS) % DEP], ((n - WS_ISS) / DEP) & 1, S_WAIT);
    }
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// Ht[n][m] = H[m][n], 32 x 32 complex tiles through shared memory
__global__ void __launch_bounds__(256) sense_transpose_kernel(const float2* __restrict__ H, int M, long long Nf,
                                                              float2* __restrict__ Ht) {
  __shared__ float2 tile[32][33];
  const long long n0 = (long long)blockIdx.x * 32;
  const int m0 = blockIdx.y * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int i = ty; i < 32; i += 8) {
    const int m = m0 + i;
    const long long n = n0 + tx;
    if (m < M && n < Nf) tile[i][tx] = H[(long long)m * Nf + n];
  }
  __syncthreads();
  for (int i = ty; i < 32; i += 8) {
    const long long n = n0 + i;
    const int m = m0 + tx;
    if (m < M && n < Nf) Ht[n * M + m] = tile[tx][i];
  }
}

// rows of the tiled matrix in row order.  Bound by memory: four rows a thread keep enough loads in flight (256
// receivers, 256^2: 91 -> 53 us a call, what a device copy of a row-major H takes; a thread moved one 8-byte value before)
constexpr int UT_ROWS = 4;
__global__ void __launch_bounds__(256) sense_untile_kernel(const float* __restrict__ in, long long rows, long long width,
                                                           long long row0, long long nrows, float* __restrict__ out) {
  const long long kp = tile_kp(width), k = 4 * ((long long)blockIdx.x * 256 + threadIdx.x);
  if (k >= width) return;
  const bool wide = ((uintptr_t)out & 15) == 0;  // (complex64 arrays need only 8; rows are multiples of 16 bytes)
  for (long long i = (long long)blockIdx.y * UT_ROWS; i < nrows; i += (long long)gridDim.y * UT_ROWS) {
    float4 v[UT_ROWS];
#pragma unroll
    for (int r = 0; r < UT_ROWS; ++r)
      if (i + r < nrows) v[r] = __ldg(reinterpret_cast<const float4*>(in + tile_off(row0 + i + r, k, rows, kp)));
#pragma unroll
    for (int r = 0; r < UT_ROWS; ++r) {
      if (i + r >= nrows) break;
      float* o = out + (i + r) * width + k;
      if (wide) {
        *reinterpret_cast<float4*>(o) = v[r];
      } else {
        reinterpret_cast<float2*>(o)[0] = make_float2(v[r].x, v[r].y);
        reinterpret_cast<float2*>(o)[1] = make_float2(v[r].z, v[r].w);
      }
    }
  }
}
// tiled Ht[n][m] = H[m][n] from tiled H, 32 x 32 complex blocks through shared memory
__global__ void __launch_bounds__(256) sense_tile_transpose_kernel(const float* __restrict__ H, int M, long long Nf,
                                                                   float* __restrict__ Ht) {
  __shared__ float2 tile[32][33];
  const long long n0 = (long long)blockIdx.x * 32, kh = tile_kp(2 * Nf), kt = tile_kp(2 * (long long)M);
  const int m0 = blockIdx.y * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int i = ty; i < 32; i += 8) {
    const int m = m0 + i;
    const long long n = n0 + tx;
    tile[i][tx] = m < M && n < Nf ? *reinterpret_cast<const float2*>(H + tile_off(m, 2 * n, M, kh)) : make_float2(0.f, 0.f);
  }
  __syncthreads();
  for (int i = ty; i < 32; i += 8) {
    const long long n = n0 + i;
    const int m = m0 + tx;
    if (2 * m < kt && n < Nf) *reinterpret_cast<float2*>(Ht + tile_off(n, 2 * m, Nf, kt)) = tile[tx][i];
  }
}

// ------------------------------------------------------------------ host side
bool sense_tc_ok(const cisor_ctx* c) {
  // 16-byte rows of H and Ht (2 Nf and 2 M floats), 2T accumulator columns <= 256
  return c->T <= 128 && c->Nf % 2 == 0 && c->M % 2 == 0;
}
bool sense_tiled(const cisor_ctx* c) { return sense_tc_ok(c) && sense_tc_cols(c->T) <= WS_NB; }
// bytes of H (rows = M of length Nf) or Ht (the other way round)
size_t sense_h_bytes(const cisor_ctx* c, long long rows, long long length) {
  return sense_tiled(c) ? sizeof(float) * (size_t)(rows * tile_kp(2 * length)) : sizeof(float2) * (size_t)rows * length;
}

// the warp-specialised kernel for nb <= 192 accumulator columns (sense_tc_cols)
using ws_fn = void (*)(const float*, long long, int, int, long long, long long, const float2*, long long, const float2*,
                       long long, int, int, long long, float2*, float2*, int*);
template <int ADJ, bool NARROW>
static ws_fn ws_kernel_of(int nb) {
  switch (nb) {
    case 32: return sense_ws_kernel<ADJ, 32, NARROW>;
    case 64: return sense_ws_kernel<ADJ, 64, NARROW>;
    case 96: return sense_ws_kernel<ADJ, 96, NARROW>;
    case 128: return sense_ws_kernel<ADJ, 128, NARROW>;
    default: return sense_ws_kernel<ADJ, 192, NARROW>;
  }
}
// for rows of K floats
template <int ADJ>
static ws_fn ws_kernel_for(int nb, long long K) {
  return tile_kp(K) % SK ? ws_kernel_of<ADJ, true>(nb) : ws_kernel_of<ADJ, false>(nb);
}

// kernel attributes (shared memory, carveout) and, for more transmitters than the warp-specialised kernel takes, the
// forward kernel's resident CTAs per SM
cisor_status sense_tc_setup(cisor_ctx* c) {
  const int nb = sense_tc_cols(c->T);
  c->sense_tc_occ = 1;
  if (sense_tiled(c)) {
    for (const void* fn : {(const void*)ws_kernel_for<0>(nb, 2 * c->Nf), (const void*)ws_kernel_for<1>(nb, 2 * (long long)c->M)})
      CISOR_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, ws_smem(nb)));
    return CISOR_OK;
  }
  for (const void* fn : {(const void*)sense_tc_kernel<0>, (const void*)sense_tc_kernel<1>}) {
    CISOR_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM));
    CISOR_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
  }
  int occ = 0;
  CISOR_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, sense_tc_kernel<0>, STH, TC_SMEM));
  c->sense_tc_occ = occ < 1 ? 1 : occ;
  return CISOR_OK;
}
// splits of the forward GEMM's K (2 Nf floats): at least one wave of resident CTAs, at most S_KMAX floats each;
// *KS = floats per split (a multiple of SK)
int sense_tc_splits(const cisor_ctx* c, long long* KS) {
  const long long K = 2 * c->Nf;
  const int mt = (c->M + 127) / 128;
  int S = c->sense_tc_occ * c->sms / mt;
  if (S < 1) S = 1;
  long long ks = ((K + S - 1) / S + SK - 1) / SK * SK;
  // below four chunks the reduction over more partials costs more than the CTAs save: 32 transmitters, 128 receivers,
  // 64^2 17.7 us with two, 15.4 with four, 16.9 with eight; 48, 130, 46^2 17.4, 16.9, 18.8
  if (sense_tiled(c) && ks < 4 * SK) ks = 4 * SK;
  if (ks > S_KMAX) ks = S_KMAX;
  if ((K + ks - 1) / ks > S_MAX) ks = ((K + S_MAX - 1) / S_MAX + SK - 1) / SK * SK;  // bounds the partials
  if (KS) *KS = ks;
  return (int)((K + ks - 1) / ks);
}

SenseTable sense_table(const cisor_ctx* c) { return {c->H, c->M, c->Nf, sense_tiled(c) ? tile_kp(2 * c->Nf) : 0}; }
// Ht from H
cisor_status sense_tc_prepare(cisor_ctx* c) {
  if (!c->Ht) return CISOR_OK;
  if (sense_tiled(c)) {
    const dim3 g((unsigned)((c->Nf + 31) / 32), (unsigned)((tile_kp(2 * (long long)c->M) / 2 + 31) / 32));
    sense_tile_transpose_kernel<<<g, 256, 0, c->stream>>>(reinterpret_cast<const float*>(c->H), c->M, c->Nf,
                                                          reinterpret_cast<float*>(c->Ht));
  } else {
    const dim3 g((unsigned)((c->Nf + 31) / 32), (unsigned)((c->M + 31) / 32));
    sense_transpose_kernel<<<g, 256, 0, c->stream>>>(c->H, c->M, c->Nf, c->Ht);
  }
  CISOR_CUDA(cudaGetLastError());
  return CISOR_OK;
}

// rows row0 .. of H, row-major, to device memory
cisor_status sense_h_rows(cisor_ctx* c, long long row0, long long nrows, float2* out) {
  if (!sense_tiled(c)) {
    CISOR_CUDA(cudaMemcpyAsync(out, c->H + row0 * c->Nf, sizeof(float2) * (size_t)nrows * c->Nf,
                               cudaMemcpyDeviceToDevice, c->stream));
    return CISOR_OK;
  }
  const long long gy = (nrows + UT_ROWS - 1) / UT_ROWS;
  sense_untile_kernel<<<dim3((unsigned)((c->Nf + 511) / 512), (unsigned)(gy < 4096 ? gy : 4096)), 256, 0, c->stream>>>(
      reinterpret_cast<const float*>(c->H), c->M, 2 * c->Nf, row0, nrows, reinterpret_cast<float*>(out));
  CISOR_CUDA(cudaGetLastError());
  c->launches += 1;
  return CISOR_OK;
}

// the GEMM over `rows` rows of the big operand (the context's widest kernel, or the one for fewer transmitters)
template <int ADJ>
static cisor_status sense_tc_gemm(cisor_ctx* c, long long rows, long long K, long long KS, int splits,
                                  const float2* src, long long lds, const float2* f, int ntx, float2* out0,
                                  float2* out1) {
  const int rtiles = (int)((rows + 127) / 128);
  c->tc_used = true;
  const float* A = reinterpret_cast<const float*>(ADJ ? c->Ht : c->H);
  if (sense_tiled(c)) {
    const int nb = sense_tc_cols(c->T), nitems = rtiles * splits;  // (the attributes were set for T's width)
    ws_kernel_for<ADJ>(nb, K)<<<nitems < c->sms ? nitems : c->sms, ws_threads(nb), ws_smem(nb), c->stream>>>(
        A, rows, rtiles, nitems, K, KS, src, lds, f, c->N, ntx, c->M, c->Nf,
        out0, out1, c->tc_err);
  } else {
    sense_tc_kernel<ADJ><<<dim3((unsigned)rtiles, (unsigned)splits), STH, TC_SMEM, c->stream>>>(
        A, K, rows, K, KS, src, lds, f, c->N, ntx, c->M, c->Nf, out0,
        out1, c->tc_err);
  }
  CISOR_CUDA(cudaGetLastError());
  return CISOR_OK;
}

// partials of Y = H (f .* u) for ntx transmitters into c->sense_part; *splits receives their count
cisor_status sense_tc_forward(cisor_ctx* c, const float2* f, const float2* u, int ntx, int* splits) {
  long long KS = 0;
  *splits = sense_tc_splits(c, &KS);
  return sense_tc_gemm<0>(c, c->M, 2 * c->Nf, KS, *splits, u, c->Nf, f, ntx, c->sense_part, nullptr);
}

// z = H^H w and b = conj(f) .* z (b may be null) for ntx transmitters
cisor_status sense_tc_adjoint(cisor_ctx* c, const float2* f, const float2* w, float2* z, float2* b, int ntx) {
  return sense_tc_gemm<1>(c, c->Nf, 2 * (long long)c->M, 2 * (long long)c->M, 1, w, c->M, f, ntx, z, b);
}

// after a call that ran the kernels above: an error if one of their waits on the tensor cores gave up.  The
// flag lives in mapped host memory, so reading it needs no synchronisation: synced = true when the call has
// already waited for its stream (every kernel it launched has finished), else the flag stays armed and the next
// call that synchronises reports a timeout of this one.
cisor_status sense_tc_check(cisor_ctx* c, bool synced) {
  if (!c->tc_used) return CISOR_OK;
  volatile int* flag = c->h_tc_err;
  if (*flag) {
    *flag = 0;
    c->tc_used = false;
    set_error("sensing: a wait on the tensor cores timed out; the outputs of this or an earlier call are invalid");
    return CISOR_ERR_CUDA;
  }
  if (synced) c->tc_used = false;
  return CISOR_OK;
}

}  // namespace cisor

// ------------------------------------------------------------------ self-test of the bounded waits
namespace cisor {
// One CTA: warp 0 takes 32 TMEM columns, every thread waits at most `polls` polls on an mbarrier that thread 0
// arrives on (arrive = 1) or that nothing completes (arrive = 0), the CTA agrees on the outcome, frees its
// tensor memory and writes 1 (completed) or 0 (gave up) to *out.  The path every tensor-core kernel above
// takes when its MMAs do not complete, without an MMA: nothing faults or hangs.
__global__ void __launch_bounds__(128) tc_wait_selftest_kernel(int arrive, int polls, int* __restrict__ out) {
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tslot;
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) mbar_init(&mbar);
  if (warp == 0) tmem_alloc(&tslot, 32);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (arrive && threadIdx.x == 0)
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&mbar)) : "memory");
  const bool ok = mbar_wait(&mbar, 0, polls);
  const bool all = !__syncthreads_or(!ok);
  if (threadIdx.x == 0) *out = all ? 1 : 0;
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tslot, 32);
}
}  // namespace cisor

extern "C" cisor_status cisor_tc_wait_selftest(int arrive, int polls, int* completed) {
  using namespace cisor;
  if (!completed || polls < 1) {
    set_error("cisor_tc_wait_selftest: NULL output or polls < 1");
    return CISOR_ERR_INVALID_ARG;
  }
  int* d = nullptr;
  CISOR_CUDA(cudaMalloc(&d, sizeof(int)));
  cudaError_t e = cudaMemset(d, 0xff, sizeof(int));
  if (e == cudaSuccess) {
    tc_wait_selftest_kernel<<<1, 128>>>(arrive ? 1 : 0, polls, d);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(completed, d, sizeof(int), cudaMemcpyDeviceToHost);
  cudaFree(d);
  if (e != cudaSuccess) return cuda_fail(e, "cisor_tc_wait_selftest", __FILE__, __LINE__);
  return CISOR_OK;
}
