"""The multiply-shift quotients of the tile geometry (csrc/geom.cuh) against
plain divisions, on the host: FastDiv over its range, the FP32 quotients of
box_index with the error of the approximate division added, and the covering
tiles of every position of small grids."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2604_16590_gb300", "csrc")

PROGRAM = r"""
#include <math.h>
#include <initializer_list>
#include <stdio.h>
#include <string.h>
#include "geom.cuh"
using namespace gattn;
static uint32_t seed = 1;
static uint32_t rnd() { return seed = seed * 1664525u + 1013904223u, (seed >> 1) ^ (seed >> 17); }
#define CHECK(c, ...) do { if (!(c)) { printf(__VA_ARGS__); return 1; } } while (0)

static int fastdiv() {
  for (int t = 0; t < 100000; ++t) {
    uint32_t d = (rnd() & 0x7fffffffu) >> (rnd() % 31);
    if (t < 300) d = t + 1;
    if (!d) d = 1;
    const FastDiv f = make_fastdiv(d);
    const uint32_t top = 0x7fffffffu, k = top / d;
    const uint32_t ns[] = {0, d - 1, d, d + 1, k * d, k * d - 1, top, top - 1, (rnd() & top) >> (rnd() % 31)};
    for (uint32_t n : ns)
      if (n <= top) CHECK((uint32_t)fdiv((int)n, f) == n / d, "fdiv %u / %u\n", n, d);
  }
  return 0;
}

// the device form of box_index: any result within two units in the last place
static int quotients() {
  for (int t = 0; t < 400000; ++t) {
    const int nb = 1 + (int)(rnd() >> (rnd() % 24 + 6)) % (1 << 20), j = (int)(rnd() % (1u << 20));
    const int js[] = {j, j / nb * nb, j / nb * nb + nb - 1};
    for (int n : js) {
      if (n >= (1 << 20)) continue;
      float q = ((float)n + 0.5f) / (float)nb;
      float lo = nextafterf(nextafterf(q, -1.f), -1.f), hi = nextafterf(nextafterf(q, 1e30f), 1e30f);
      CHECK((int)lo == n / nb && (int)hi == n / nb, "quotient %d / %d\n", n, nb);
    }
  }
  return 0;
}

static int covers(int G, int c, int h) {
  Geom g;
  memset(&g, 0, sizeof(g));
  const int n = (G + c - 1) / c;
  for (int a = 0; a < 3; ++a) {
    g.G[a] = a == 1 ? G : 1;
    g.c[a] = a == 1 ? c : 1;
    g.h[a] = a == 1 ? h : 0;
    g.n[a] = a == 1 ? n : 1;
    g.fc[a] = make_fastdiv(g.c[a]);
    g.fG[a] = make_fastdiv(g.G[a]);
  }
  g.N = G;
  g.ntiles = n;
  g.fN = make_fastdiv(G);
  g.fn2 = make_fastdiv(1);
  g.fn12 = make_fastdiv(n);
  for (int p = 0; p < G; ++p) {
    int first = -1, last = -1;
    for (int k = 0; k < n; ++k) {
      TileBox tb;
      tile_box(g, k, tb);
      CHECK(tb.k[1] == k && tb.lo[1] == (k * c - h > 0 ? k * c - h : 0), "tile_box %d\n", k);
      if (p >= tb.lo[1] && p < tb.lo[1] + tb.e[1]) {
        if (first < 0) first = k;
        last = k;
      }
    }
    int k0, k1;
    cover_dim(g, 1, p, k0, k1);
    CHECK(k0 == first && k1 == last, "cover G %d c %d h %d p %d\n", G, c, h, p);
    const int pos[3] = {0, p, 0};
    for (int k = first; k <= last; ++k) {
      TileBox tb;
      tile_box(g, k, tb);
      CHECK(only_cover(g, tb, pos) == (first == last), "only_cover G %d c %d h %d p %d\n", G, c, h, p);
    }
  }
  return 0;
}

static int rows() {  // batch*head and token of a row index, on both sides of 2^31
  const int64_t Ns[] = {1, 7, 262144, 1000003, (1LL << 31) - 1};
  for (int64_t N : Ns) {
    Geom g;
    memset(&g, 0, sizeof(g));
    g.N = N;
    g.fN = make_fastdiv((uint32_t)N);
    for (int64_t bh : {0, 1, 3, 2147, 2148, 65534})
      for (int64_t i : {(int64_t)0, N / 2, N - 1}) {
        int b;
        int64_t k;
        split_row(g, bh * N + i, b, k);
        CHECK(b == bh && k == i, "split_row N %lld bh %lld\n", (long long)N, (long long)bh);
      }
  }
  return 0;
}

int main() {
  if (fastdiv() || quotients() || rows()) return 1;
  for (int G = 1; G <= 40; ++G)
    for (int c = 1; c <= 12; ++c)
      for (int h = 0; h <= 14; ++h)
        if (covers(G, c, h)) return 1;
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("geom")
    src, exe = d / "geom.cpp", d / "geom"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)],
                   check=True)
    return str(exe)


def test_quotients_and_covers_match_plain_divisions(program):
    r = subprocess.run([program], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
