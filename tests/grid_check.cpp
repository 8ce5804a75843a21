// The scene-grid 4-wide nodes on the host: same tree as the 8-bit nodes, boxes
// that contain the triangles below them, and a float emulation of the
// traversal's plane arithmetic that never misses a box the exact ray meets.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <functional>
#include <random>
#include <string>
#include <vector>

#include "ipt_internal.h"

static float as_float(uint32_t w) {
  float f;
  std::memcpy(&f, &w, 4);
  return f;
}

struct Axis {
  float A, Bn, Bf;
  bool neg;
};

static Axis axis(float lo, float s, float o, float d) {
  const float tiny = 1e-30f;
  const float inv = 1.0f / (std::fabs(d) > tiny ? d : std::copysign(tiny, d));
  Axis a;
  a.A = s * inv;
  const float C = (lo - o) * inv, B = std::fmaf(lo - o, inv, -a.A);
  const float m = 0x1p-21f * (std::fabs(a.A) + std::fabs(C));
  a.Bn = B - m;
  a.Bf = B + m;
  a.neg = inv < 0.0f;
  return a;
}

static float unit(uint32_t plane) { return as_float(0x3F000000u | (plane << 8)); }

static int check(const char* name, const std::vector<float>& pos, bool want_grid) {
  const uint32_t nt = (uint32_t)(pos.size() / 9);
  std::vector<uint32_t> idx(3 * nt), seg(nt, 0);
  for (uint32_t i = 0; i < 3 * nt; ++i) idx[i] = i;
  ipt::HostScene s;
  std::string err;
  if (!ipt::build_scene(pos.data(), 3 * nt, nullptr, idx.data(), nt, seg.data(), 1, &s, &err)) {
    std::printf("%s: %s\n", name, err.c_str());
    return 1;
  }
  if (s.nodes4g.empty() == want_grid) {
    std::printf("%s: scene grid %s\n", name, want_grid ? "missing" : "not expected");
    return 1;
  }
  if (s.nodes4g.empty()) return 0;
  const auto plane = [&](int a, uint32_t q) { return (double)s.grid_lo[a] + (q & 0x7FFFu) * ((double)s.grid_s[a] / 32768.0); };
  int bad = 0;
  // bounds of every subtree against its box
  std::function<void(int, double*, double*)> bounds = [&](int ref, double* lo, double* hi) {
    for (int a = 0; a < 3; ++a) lo[a] = 1e300, hi[a] = -1e300;
    if (ref < 0) {
      const int v = -ref - 1;
      for (int i = v >> 3; i < (v >> 3) + (v & 7) + 1; ++i)
        for (int k = 0; k < 9; ++k) {
          const double x = s.tris[12 * (size_t)i + 4 * (k / 3) + k % 3];
          lo[k % 3] = std::min(lo[k % 3], x);
          hi[k % 3] = std::max(hi[k % 3], x);
        }
      return;
    }
    const uint32_t *g = &s.nodes4g[16 * (size_t)ref], *l = &s.nodes4[16 * (size_t)ref];
    for (int i = 0; i < 4; ++i) {
      if (g[12 + i] != l[4 + i]) ++bad;
      if ((g[i] & 0xFFFFu) > (g[i] >> 16)) continue;  // empty slot: inverted
      double cl[3], ch[3];
      bounds((int)g[12 + i], cl, ch);
      for (int a = 0; a < 3; ++a) {
        if (plane(a, g[4 * a + i]) > cl[a] || plane(a, g[4 * a + i] >> 16) < ch[a]) ++bad;
        lo[a] = std::min(lo[a], cl[a]);
        hi[a] = std::max(hi[a], ch[a]);
      }
    }
  };
  double lo[3], hi[3];
  bounds(0, lo, hi);
  if (bad) {
    std::printf("%s: %d links or boxes wrong\n", name, bad);
    return 1;
  }
  // rays aimed at points on the boxes' faces, edges and corners
  std::mt19937 rng(5);
  std::uniform_real_distribution<double> un(0.0, 1.0);
  const size_t nodes = s.nodes4g.size() / 16;
  for (int it = 0; it < 200000; ++it) {
    const uint32_t* g = &s.nodes4g[16 * (rng() % nodes)];
    const int i = rng() % 4;
    if ((g[i] & 0xFFFFu) > (g[i] >> 16)) continue;
    double bl[3], bh[3];
    float o[3], d[3];
    const double away = it % 7 == 0 ? 300.0 : (it % 2 ? 1.0 : 0.05);
    for (int a = 0; a < 3; ++a) {
      bl[a] = plane(a, g[4 * a + i]);
      bh[a] = plane(a, g[4 * a + i] >> 16);
      const int pick = rng() % 4;
      const double p = pick == 0 ? bl[a] : (pick == 1 ? bh[a] : bl[a] + un(rng) * (bh[a] - bl[a]));
      o[a] = (float)(p + (un(rng) - 0.5) * away * (hi[a] - lo[a] + 1e-3));
      d[a] = (float)(p - o[a]);
      if (rng() % 6 == 0) o[a] = (float)p, d[a] = rng() % 2 ? 0.0f : -0.0f;  // parallel to a face plane
    }
    if (d[0] == 0.0f && d[1] == 0.0f && d[2] == 0.0f) continue;
    // exact slab test (a zero component: inside the slab or a miss)
    long double n = 0.0L, f = HUGE_VALL;
    bool miss = false;
    for (int a = 0; a < 3; ++a) {
      if (d[a] == 0.0f) {
        miss = miss || o[a] < bl[a] || o[a] > bh[a];
        continue;
      }
      long double t0 = ((long double)bl[a] - o[a]) / d[a], t1 = ((long double)bh[a] - o[a]) / d[a];
      if (t0 > t1) std::swap(t0, t1);
      n = std::max(n, t0);
      f = std::min(f, t1);
    }
    if (miss || n > f) continue;
    float tn = 0.0f, tf = INFINITY;
    for (int a = 0; a < 3; ++a) {
      const Axis x = axis(s.grid_lo[a], s.grid_s[a], o[a], d[a]);
      const uint32_t pl = g[4 * a + i] & 0xFFFFu, ph = g[4 * a + i] >> 16;
      tn = std::fmax(tn, std::fmaf(unit(x.neg ? ph : pl), x.A, x.Bn));
      tf = std::fmin(tf, std::fmaf(unit(x.neg ? pl : ph), x.A, x.Bf));
    }
    if (!(tn <= tf)) ++bad;
  }
  if (bad) std::printf("%s: %d exact hits missed\n", name, bad);
  return bad ? 1 : 0;
}

int main() {
  std::mt19937 rng(3);
  std::uniform_real_distribution<float> un(-1.0f, 1.0f);
  const auto soup = [&](int n, float size, float scale, float shift) {
    std::vector<float> p;
    for (int i = 0; i < n; ++i) {
      const float c[3] = {4.0f * un(rng), 1.5f * un(rng), 3.0f * un(rng)};
      for (int k = 0; k < 9; ++k) p.push_back(scale * (c[k % 3] + size * un(rng)) + shift);
    }
    return p;
  };
  std::vector<float> flat;
  for (int i = 0; i < 2000; ++i)
    for (int k = 0; k < 9; ++k) flat.push_back(k % 3 == 1 ? 0.25f : 5.0f * un(rng));
  std::vector<float> detail = soup(3000, 0.3f, 1e-3f, 0.0f);  // a millimetre-sized object in a large room
  for (float c : {-40.0f, 40.0f})
    for (int k = 0; k < 9; ++k) detail.push_back(c + un(rng));
  int bad = 0;
  bad += check("soup", soup(3000, 0.2f, 1.0f, 0.0f), true);
  bad += check("shifted soup", soup(500, 0.2f, 1.0f, 100.0f), true);
  bad += check("two triangles", soup(2, 0.5f, 1.0f, 0.0f), true);
  bad += check("one triangle", soup(1, 0.5f, 1.0f, 0.0f), true);
  bad += check("flat", flat, true);
  bad += check("small detail", detail, false);
  bad += check("huge coordinates", soup(300, 0.2f, 1e25f, 0.0f), false);
  bad += check("tiny coordinates", soup(300, 0.2f, 1e-12f, 0.0f), false);
  return bad ? 1 : 0;
}
