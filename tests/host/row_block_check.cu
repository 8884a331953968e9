// The row-block matvec's layout (block_layout_host) and its coset arithmetic (syk_block.cuh, host
// branches) against the plain sum over masks, row by row, without a GPU.  Every offset that a thread
// would read is checked against the tile, the chunk and the table memory.
// Prints the largest relative error (2-norm) over all shapes; exits non-zero on an offset out of range.
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "syk_block.cuh"
#include "syk_internal.h"

using namespace syk;
using namespace syk::blk;
using cd = std::complex<double>;

namespace {

void require(bool ok, const char* what) {
  if (!ok) {
    std::printf("out of range: %s\n", what);
    std::exit(1);
  }
}

// y = H x as the sum over masks, from the term set's FP64 tables
std::vector<cd> plain(const syk_terms* t, int sector, const std::vector<cd>& x, int B) {
  const int n = t->n;
  std::vector<cd> y(x.size());
  for (int64_t c = 0; c < t->D; ++c) {
    const uint32_t xf = uint32_t(c) | uint32_t((__builtin_popcountll(c) + sector) & 1) << (n - 1);
    auto add = [&](cd co, uint32_t flip) {
      for (int b = 0; b < B; ++b) y[c * B + b] += co * x[(c ^ flip) * B + b];
    };
    double d = 0.0;
    for (int a = 0; a < n; ++a)
      for (int b = a + 1; b < n; ++b) d += ((xf >> a) ^ (xf >> b)) & 1 ? -t->wdiag[a * n + b] : t->wdiag[a * n + b];
    add(d, 0);
    for (int k = 0; k < t->n2; ++k) {
      const uint32_t* r = &t->m2_rec[4 * size_t(k)];
      const int u = ((xf >> (r[2] & 255)) & 1) | (((xf >> ((r[2] >> 8) & 255)) & 1) << 1);
      cd s = 0.0;
      for (int q = 0; q < n; ++q) {
        const double* w = &t->m2_tab[((size_t(k) * n + q) * 4 + u) * 2];
        s += (xf >> q) & 1 ? -cd(w[0], w[1]) : cd(w[0], w[1]);
      }
      add(__builtin_popcount(r[1] & xf) & 1 ? -s : s, r[0]);
    }
    for (int k = 0; k < t->n4; ++k) {
      const uint32_t* r = &t->m4_rec[4 * size_t(k)];
      int u = (__builtin_popcount(r[1] & xf) & 1) << 4;
      for (int q = 0; q < 4; ++q) u |= (xf >> ((r[2] >> (8 * q)) & 255)) & (1u << q);
      const double* v = &t->m4_tab[(size_t(k) * 32 + u) * 2];
      add(cd(v[0], v[1]), r[0]);
    }
  }
  return y;
}

// One launch shape: every thread of every tile walks the chunks as k_apply_block does.
template <int RB, bool LOWS>
double check(const syk_terms* t, int sector, int B, int lb, int mb, int cs, int auxb) {
  BlockHost H;
  require(block_layout_host(t, RB, lb, mb, cs, auxb, false, &H) == SYK_OK, "layout");
  const int n = t->n, SE = B << lb;
  const int64_t D = t->D, T = int64_t(1) << (lb + RB + mb);
  const size_t tile_bytes = size_t(T) * B * 8;
  std::mt19937 g(7);
  std::normal_distribution<float> nd;
  std::vector<float2> x(D * B), y(D * B, make_float2(1e30f, 0.f));
  std::vector<cd> xd(D * B);
  for (size_t i = 0; i < x.size(); ++i) {
    x[i] = make_float2(nd(g), nd(g));
    xd[i] = cd(x[i].x, x[i].y);
  }
  const std::vector<float> fd(t->wdiag.begin(), t->wdiag.end());
  for (int64_t tile = 0; tile < D / T; ++tile)
    for (int th = 0; th < (SE << mb); ++th) {
      const int mid = th / SE, e = th % SE, low = e / B, s = e % B;
      Acc<RB> a = {};
      RowCtx c = {};
      c.x = uint32_t(tile * T) | uint32_t(mid) << (lb + RB) | uint32_t(low);
      c.q = (__builtin_popcount(c.x) + sector) & 1;
      c.above = __builtin_popcount(c.x >> (lb + RB)) & 1;
      c.xn = (c.x & ((1u << lb) - 1)) | (c.x >> (lb + RB)) << lb;
      c.n = n;
      c.LB = lb;
      c.ng = (n - 1 - RB + 3) / 4;
      c.wd = fd.data();
      for (int q = H.begin[0]; q < H.begin[cs]; ++q) {
        const int4 ch = H.chunks[q];
        const size_t at = size_t(ch.y) * 16, bytes = size_t(ch.z) * 16;
        require(at + bytes <= H.blob.size() && bytes <= size_t(auxb), "chunk");
        const unsigned char* blob = H.blob.data() + at;
        const unsigned char* part = reinterpret_cast<const unsigned char*>(&x[(tile ^ ch.x) * T * B]);
        const uint4* rec = reinterpret_cast<const uint4*>(blob);
        const uint4 head = *rec++;
        auto partner = [&](const uint4 rc) {
          const size_t off = (size_t((uint32_t(mid) ^ (rc.x & 0xffff)) << RB) * SE +
                              (uint32_t(low) ^ ((rc.x >> 16) & 0xff)) * B + s) * 8;
          require(off + size_t((1 << RB) - 1) * SE * 8 + 8 <= tile_bytes, "partner row");
          return part + off;
        };
        auto run = [&](auto w, uint32_t count) {
          constexpr int W = decltype(w)::value;
          for (uint32_t k = 0; k < count; ++k) {
            const uint4 rc = *rec++;
            require(rc.w + size_t(coset_bytes(RB, W, c.ng)) <= bytes, "coset tables");
            const CosetAt k2 = {partner(rc), blob + rc.w, support(c.x, rc.z), parity(rc.y & c.x), rc.x >> 31};
            coset<RB, W, LOWS>(a, k2, SE * 8, c);
          }
        };
        run(std::integral_constant<int, 4>{}, head.x & 255);
        run(std::integral_constant<int, 3>{}, (head.x >> 8) & 255);
        run(std::integral_constant<int, 2>{}, (head.x >> 16) & 255);
        run(std::integral_constant<int, 1>{}, head.x >> 24);
        run(std::integral_constant<int, 0>{}, head.y & 255);
        for (uint32_t k = head.y >> 8; k > 0; --k) {
          const uint4 rc = *rec++;
          require(rc.w + size_t(m2_bytes(RB, c.ng)) <= bytes, "two-spin tables");
          m2_record<RB, false>(a, partner(rc), SE * 8, rc, blob + rc.w, c);
        }
      }
      for (int r = 0; r < (1 << RB); ++r) {
        const float2 re = unpack2(a.re[r]), im = unpack2(a.im[r]);
        y[size_t(tile * T + (int64_t(mid) << (lb + RB)) + (int64_t(r) << lb) + low) * B + s] =
            make_float2(re.x - im.y, re.y + im.x);
      }
    }
  const std::vector<cd> ref = plain(t, sector, xd, B);
  double num = 0.0, den = 0.0;
  for (size_t i = 0; i < ref.size(); ++i) {
    num += std::norm(cd(y[i].x, y[i].y) - ref[i]);
    den += std::norm(ref[i]);
  }
  const double err = std::sqrt(num / den);
  if (!(err < 2e-6)) std::printf("N=%d sector=%d RB=%d B=%d LB=%d MB=%d CTAs=%d: %.3g\n", t->N, sector, RB, B, lb, mb, cs, err);
  return err;
}

}  // namespace

int main() {
  double worst = 0.0;
  int shapes = 0;
  for (int N : {12, 14, 16, 18, 20}) {
    std::mt19937_64 g(N);
    std::normal_distribution<double> nd(0.0, std::sqrt(6.0 / (double(N) * N * N)));
    std::vector<double> J(size_t(N) * (N - 1) * (N - 2) * (N - 3) / 24);
    for (double& j : J) j = nd(g);
    syk_terms* t = nullptr;
    require(syk_build_terms(N, J.data(), &t) == SYK_OK, "terms");
    const int nb = t->n - 1, aux5 = coset_most(5, (nb - 5 + 3) / 4), aux3 = coset_most(3, (nb - 3 + 3) / 4);
    auto note = [&](double e) {
      worst = e > worst || e != e ? e : worst;
      ++shapes;
    };
    for (int sector : {0, 1})
      for (int lb : {0, 1, 2, 4})
        for (int mb : {0, 1, 2})
          for (int cs : {1, 3, 8}) {
            if (cs > 1 && mb != 1) continue;
            const int B = lb == 4 ? 1 : lb == 2 ? 3 : lb == 1 ? 5 : 2;
            if (lb + 5 + mb <= nb) note(check<5, true>(t, sector, B, lb, mb, cs, aux5));
            if (lb == 0 && 5 + mb <= nb) note(check<5, false>(t, sector, B, lb, mb, cs, aux5));
            if (lb + 3 + mb <= nb) note(check<3, true>(t, sector, B, lb, mb, cs, aux3));
          }
    syk_free_terms(t);
  }
  std::printf("shapes %d worst %.3g\n", shapes, worst);
  return worst < 2e-6 ? 0 : 1;
}
