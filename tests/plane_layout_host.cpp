// Host enumeration of the shared-memory accesses of the 3D plane convolution
// (csrc/plane_layout.cuh).  Prints, per FFT side and access group, the most
// lanes of a half-warp that meet one bank of 8 bytes (1: no conflict) and whether
// every value is read where it was written, in its own slot, inside the CTA's
// shared memory.
#include <cstdio>
#include <map>
#include <set>
#include <vector>

#include "plane_layout.cuh"

using namespace cisor;

static int worst;
static bool good;
static int limit;

// addresses of the 32 lanes of one access
template <class F> static void access(F f) {
  for (int h = 0; h < 2; ++h) {
    std::vector<std::set<int>> bank(16);
    for (int l = 16 * h; l < 16 * h + 16; ++l) {
      const int a = f(l);
      good = good && a >= 0 && a + 8 <= limit && a % 8 == 0;
      bank[(a / 8) % 16].insert(a);
    }
    for (auto& b : bank) worst = (int)b.size() > worst ? (int)b.size() : worst;
  }
}

template <int P> static void run() {
  typedef PlaneLayout<P> L;
  const int E = L::E, NT = L::NT, Q = L::Q, PB = L::PB, M = L::M;
  auto begin = [&](int bytes) { worst = 0; good = true; limit = bytes; };
  auto out = [&](const char* what) { printf("%d %s %d %d\n", P, what, worst, (int)good); };
  std::map<std::pair<int, int>, int> slot;  // (transform, value) -> address
  auto put = [&](int tr, int i, int a) { slot[{tr, i}] = a; };
  auto get = [&](int tr, int i, int a) { good = good && slot.count({tr, i}) && slot[{tr, i}] == a; };
  auto distinct = [&]() {
    std::set<int> s;
    for (auto& k : slot) s.insert(k.second);
    good = good && s.size() == slot.size();
    slot.clear();
  };
  // rows of the plane
  auto rlt = [](int l) { return l % 8; };
  auto rz = [](int l) { return ((l >> 3) & 1) * 2 + (l >> 4); };
  begin(L::XOFF);
  for (int z0 = 0; z0 < L::H; z0 += 4) {
    auto natural = [&](bool write) {
      for (int q = 0; q < Q; ++q)
        for (int r = 0; r < NT; ++r)
          access([&](int l) {
            const int z = z0 + rz(l), a = L::row_nat(z, rlt(l)) ^ L::row_nat_k(q, r);
            if (write) put(z, rlt(l) + NT * q + E * r, a);
            return a;
          });
    };
    for (int k = 0; k < E; ++k)
      access([&](int l) {
        const int z = z0 + rz(l), a = L::row_fw(z, rlt(l)) ^ L::row_fw_k(k);
        put(z, E * rlt(l) + k, a);
        return a;
      });
    for (int q = 0; q < Q; ++q)
      for (int r = 0; r < NT; ++r)
        access([&](int l) {
          const int z = z0 + rz(l), a = L::row_nat(z, rlt(l)) ^ L::row_fr_k(q, r);
          get(z, rlt(l) + NT * q + E * r, a);
          return a;
        });
    distinct();
    natural(true);
    distinct();
    for (int q = 0; q < Q; ++q)
      for (int s = 0; s < NT; ++s)
        access([&](int l) {
          const int z = z0 + rz(l), a = L::row_iw(z, rlt(l)) ^ L::row_iw_k(q, s);
          put(z, NT * (rlt(l) + NT * q) + s, a);
          return a;
        });
    for (int r = 0; r < E; ++r)
      access([&](int l) {
        const int z = z0 + rz(l), a = L::row_nat(z, rlt(l)) ^ L::row_ir_k(r);
        get(z, rlt(l) + NT * r, a);
        return a;
      });
    distinct();
  }
  out("rows");
  // columns
  auto cw = [](int l) { return l & 3; };
  auto clt = [](int l) { return l >> 2; };
  begin(L::BYTES);
  for (int c0 = 0; c0 < P; c0 += 4) {
    const int x0 = c0 % L::XCOLS;
    auto base = [&](bool up, int l) { return up ? L::col_rx(clt(l), x0 + cw(l)) : L::col_r(clt(l), c0 + cw(l)); };
    for (int k = 0; k < E; ++k)
      access([&](int l) {
        const int a = (L::col_fw(clt(l), c0 + cw(l), x0 + cw(l)) ^ ((k & 3) * M)) + (k >> 2) * 4 * PB;
        put(cw(l), E * clt(l) + k, a);
        return a;
      });
    for (int q = 0; q < Q; ++q)
      for (int r = 0; r < NT; ++r)
        access([&](int l) {
          const int a = (base(L::fr_up(r), l) ^ ((r & 3) * M)) + L::fr_off(q, r);
          get(cw(l), clt(l) + NT * q + E * r, a);
          return a;
        });
    distinct();
    for (int q = 0; q < Q; ++q)
      for (int s = 0; s < NT; ++s)
        access([&](int l) {
          const int a = (L::col_iw(clt(l), q, c0 + cw(l), x0 + cw(l)) ^ ((s & 3) * M)) + (s >> 2) * 4 * PB;
          put(cw(l), NT * (clt(l) + NT * q) + s, a);
          return a;
        });
    for (int r = 0; r < E; ++r)
      access([&](int l) {
        const int a = (base(L::ir_up(r), l) ^ ((r & 3) * M)) + L::ir_off(r);
        get(cw(l), clt(l) + NT * r, a);
        return a;
      });
    distinct();
    // natural order is the one the rows use
    for (int k = 0; k < E / 2; ++k)
      access([&](int l) {
        const int z = clt(l) + NT * k, ky = c0 + cw(l), a = L::col_r(clt(l), ky) + NT * k * PB;
        good = good && a == (L::row_nat(z, ky % 8) ^ L::row_nat_k((ky % E) / 8, ky / E));
        return a;
      });
  }
  // a warp's exchange stays in its own columns of the plane and of xs
  for (int c0 = 0; c0 < L::XCOLS; c0 += 4)
    for (int l = 0; l < 32; ++l)
      for (int row = 0; row < L::H; ++row) {
        put(c0 / 4, 64 * row + cw(l), L::part(row, c0 + cw(l), row & 3));
        put(c0 / 4, 8192 + 64 * row + cw(l), L::xpart(row, c0 + cw(l), row & 3));
      }
  distinct();
  out("columns");
  // the row kernels' exchange
  begin(P * 32 * 8);
  for (int w = 0; w < 8; ++w) {
    for (int k = 0; k < E; ++k)
      access([&](int l) {
        const int a = L::rk_fw(l % 8, 4 * w + l / 8) + 256 * k;
        put(4 * w + l / 8, E * (l % 8) + k, a);
        return a;
      });
  }
  for (int lt = 0; lt < NT; ++lt)
    for (int q = 0; q < Q; ++q)
      for (int r = 0; r < NT; ++r)
        access([&](int l) {
          const int a = L::rk_fr(lt, l, r) + 2048 * q;
          get(l, lt + NT * q + E * r, a);
          return a;
        });
  distinct();
  for (int lt = 0; lt < NT; ++lt)
    for (int q = 0; q < Q; ++q)
      for (int s = 0; s < NT; ++s)
        access([&](int l) {
          const int a = L::rk_iw(lt, l, s) + 16384 * q;
          put(l, NT * (lt + NT * q) + s, a);
          return a;
        });
  for (int w = 0; w < 8; ++w)
    for (int r = 0; r < E; ++r)
      access([&](int l) {
        const int a = L::rk_ir(l % 8, 4 * w + l / 8) + 2048 * r;
        get(4 * w + l / 8, l % 8 + NT * r, a);
        return a;
      });
  distinct();
  out("row_kernels");
  // twiddles: 8 lanes of a row or column, the other lanes repeat them
  begin(L::TW * 8);
  for (int q = 0; q < Q; ++q)
    for (int r = 0; r < NT; ++r) access([&](int l) { return 8 * L::tw(r, l % 8 + NT * q); });
  for (int r = 0; r < E; ++r) access([&](int l) { return 8 * L::tw(l % 8, r); });
  out("twiddles");
}

int main() {
  run<64>();
  run<128>();
}
