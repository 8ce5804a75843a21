// Rays from far away against the 4-wide nodes: where the node's own 8-bit grid
// rejects an empty slot (an inverted box), the scene grid rejects it too, so a
// ray that missed does not come to walk the root again and again.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "ipt_internal.h"

static float as_float(uint32_t w) {
  float f;
  std::memcpy(&f, &w, 4);
  return f;
}

struct Ray {
  float o[3], inv[3];
};

// The slab tests of node4_children and node4g_children for slot i.
static bool hit8(const uint32_t* w, int i, const Ray& r) {
  const float scale[3] = {as_float(w[3]), as_float(w[14]), as_float(w[15])};
  const auto unit = [](uint32_t q) { return as_float(0x3F800000u | (q << 8)); };
  float tn = 0.0f, tf = INFINITY;
  for (int a = 0; a < 3; ++a) {
    const float A = scale[a] * r.inv[a], B = std::fmaf(as_float(w[a]) - r.o[a], r.inv[a], -A);
    const uint32_t lo = (w[8 + 2 * a] >> (8 * i)) & 255u, hi = (w[9 + 2 * a] >> (8 * i)) & 255u;
    const bool neg = r.inv[a] < 0.0f;
    tn = std::fmax(tn, std::fmaf(unit(neg ? hi : lo), A, std::fmaf(std::fabs(A), -0x1p-22f, B)));
    tf = std::fmin(tf, std::fmaf(unit(neg ? lo : hi), A, std::fmaf(std::fabs(A), 0x1p-22f, B)));
  }
  return tn <= tf * 1.0000005f;
}

static bool hit_grid(const ipt::HostScene& s, const uint32_t* g, int i, const Ray& r) {
  const auto unit = [](uint32_t plane) { return as_float(0x3F000000u | (plane << 8)); };
  float tn = 0.0f, tf = INFINITY;
  for (int a = 0; a < 3; ++a) {
    const float A = s.grid_s[a] * r.inv[a], C = (s.grid_lo[a] - r.o[a]) * r.inv[a];
    const float B = std::fmaf(s.grid_lo[a] - r.o[a], r.inv[a], -A);
    const float m = std::fmin(0x1p-21f * (std::fabs(A) + std::fabs(C)), 0x1.fffffep127f);
    const uint32_t lo = g[4 * a + i] & 0xFFFFu, hi = g[4 * a + i] >> 16;
    const bool neg = r.inv[a] < 0.0f;
    tn = std::fmax(tn, std::fmaf(unit(neg ? hi : lo), A, B - m));
    tf = std::fmin(tf, std::fmaf(unit(neg ? lo : hi), A, B + m));
  }
  return tn <= tf && tn < INFINITY;
}

int main() {
  std::mt19937 rng(3);
  std::uniform_real_distribution<float> un(-1.0f, 1.0f);
  const uint32_t nt = 3000;
  std::vector<float> pos;
  for (uint32_t i = 0; i < nt; ++i) {
    const float c[3] = {4.0f * un(rng), 1.5f * un(rng), 3.0f * un(rng)};
    for (int k = 0; k < 9; ++k) pos.push_back(c[k % 3] + 0.2f * un(rng));
  }
  std::vector<uint32_t> idx(3 * nt), seg(nt, 0);
  for (uint32_t i = 0; i < 3 * nt; ++i) idx[i] = i;
  ipt::HostScene s;
  std::string err;
  if (!ipt::build_scene(pos.data(), 3 * nt, nullptr, idx.data(), nt, seg.data(), 1, &s, &err) || s.nodes4g.empty())
    return 1;
  std::vector<std::pair<int, int>> empty;  // (node, slot)
  for (size_t n = 0; n < s.nodes4g.size() / 16; ++n)
    for (int i = 0; i < 4; ++i)
      if ((s.nodes4g[16 * n + i] & 0xFFFFu) > (s.nodes4g[16 * n + i] >> 16)) empty.push_back({(int)n, i});
  int bad = 0;
  for (double dist : {10.0, 1e3, 1e6, 1e7, 1e9, 1e20, 1e30, 2e38, (double)INFINITY})
    for (int it = 0; it < 20000; ++it) {
      Ray r;
      double u[3], d[3], len = 0.0;
      for (int a = 0; a < 3; ++a) u[a] = un(rng), len += u[a] * u[a];
      const int kind = it % 3;  // any direction, towards the scene's middle, none
      for (int a = 0; a < 3; ++a) {
        r.o[a] = (float)(dist * (u[a] / std::sqrt(len)));
        d[a] = kind == 0 ? un(rng) : (kind == 1 ? -u[a] : 0.0);
        const float f = (float)d[a], tiny = 1e-30f;
        r.inv[a] = 1.0f / (std::fabs(f) > tiny ? f : std::copysign(tiny, f));
      }
      const auto [n, i] = empty[rng() % empty.size()];
      if (!hit8(&s.nodes4[16 * (size_t)n], i, r) && hit_grid(s, &s.nodes4g[16 * (size_t)n], i, r)) ++bad;
    }
  if (bad) std::printf("%d empty slots entered\n", bad);
  return bad ? 1 : 0;
}
