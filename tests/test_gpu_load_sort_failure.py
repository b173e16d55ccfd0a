"""When a sort of a load reports that its grid barrier gave up, the kernels behind it do nothing.

The rows are then in any order or partly unwritten, so nothing may be indexed by them.  A harness
compiled with hm_graph.cu launches each of these kernels on small valid rows (so that every access
is in range whether or not a kernel looks at the word), once with the word set -- every output must
keep its filling -- and once without, where every output must change.
"""
from __future__ import annotations

import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

_HARNESS = r"""
#include "hm_graph.cu"
#include <cstdio>

int main() {
  // vertex v -> v + 1 .. v + 40 (mod n): sorted by source, and 2,048 rows of one hub for k_group_hubs
  const int n = 4096, deg = 40;
  std::vector<int4> rows;
  for (int v = 0; v < n; ++v) {
    const int d = v == 7 ? 2048 : deg;
    std::vector<int> to;
    for (int i = 1; i <= d; ++i) to.push_back((v + i) % n);
    std::sort(to.begin(), to.end());
    for (int w : to) rows.push_back(make_int4(v, w, w & 1, 0));
  }
  const int64_t m = (int64_t)rows.size();
  const Classes C{4, 2, 0, 0};
  std::vector<int32_t> vlab(n);
  for (int v = 0; v < n; ++v) vlab[v] = v & 1;
  const uint32_t nword = (uint32_t)(4 * ((m + 7) / 8)), nbkt = (uint32_t)m;
  const int64_t rwords = (m >> 1) + n + 1;
  struct Out { const char *name; size_t bytes; unsigned char *p; };
  std::vector<Out> outs = {{"src", 4 * (size_t)m}, {"adj", 4 * (size_t)m}, {"lab", 4 * (size_t)m}, {"off", 8 * (size_t)(n + 1)},
                           {"filter", 8 * (size_t)nword}, {"regions", 8 * (size_t)rwords}, {"hash", 32 * (size_t)nbkt},
                           {"gadj", 4 * (size_t)m}, {"gofs", 4 * ((size_t)n * 4 + 1)}, {"ngroup", 4 * (size_t)(n + 1)},
                           {"hubs", 4 * (size_t)(m / kHub + 1)}, {"gadj of the hub", 4 * (size_t)m}};
  for (Out &o : outs) cudaMalloc((void **)&o.p, o.bytes);
  int4 *d_rows;
  int32_t *d_vlab, *fixed_adj, *fixed_lab, *d_hub;
  int64_t *fixed_off;
  uint32_t *word;  // {input errors, sort error, long lists}
  cudaMalloc((void **)&d_rows, 16 * m);
  cudaMalloc((void **)&d_vlab, 4 * n);
  cudaMalloc((void **)&fixed_adj, 4 * m);
  cudaMalloc((void **)&fixed_lab, 4 * m);
  cudaMalloc((void **)&fixed_off, 8 * (n + 1));
  cudaMalloc((void **)&d_hub, 8);
  cudaMalloc((void **)&word, 16);
  cudaMemcpy(d_rows, rows.data(), 16 * m, cudaMemcpyHostToDevice);
  cudaMemcpy(d_vlab, vlab.data(), 4 * n, cudaMemcpyHostToDevice);
  std::vector<int32_t> adj(m), lab(m);
  std::vector<int64_t> off(n + 1, 0);
  for (int64_t e = 0; e < m; ++e) {
    adj[e] = rows[e].y;
    lab[e] = rows[e].z;
    off[rows[e].x + 1] = e + 1;
  }
  cudaMemcpy(fixed_adj, adj.data(), 4 * m, cudaMemcpyHostToDevice);
  cudaMemcpy(fixed_lab, lab.data(), 4 * m, cudaMemcpyHostToDevice);
  cudaMemcpy(fixed_off, off.data(), 8 * (n + 1), cudaMemcpyHostToDevice);
  const int32_t hub[2] = {7, 1};
  cudaMemcpy(d_hub, hub, 8, cudaMemcpyHostToDevice);
  int bad = 0;
  for (uint32_t failed = 0; failed < 2; ++failed) {
    for (Out &o : outs) cudaMemset(o.p, o.p == outs[6].p ? 0xff : o.p == outs[4].p || o.p == outs[5].p ? 0 : 0x5a, o.bytes);
    const uint32_t w[4] = {0, failed, 0, 0};
    cudaMemcpy(word, w, 16, cudaMemcpyHostToDevice);
    const int *err = reinterpret_cast<const int *>(word + 1);
    auto as32 = [&](int i) { return reinterpret_cast<int32_t *>(outs[i].p); };
    auto as64 = [&](int i) { return reinterpret_cast<unsigned long long *>(outs[i].p); };
    uint32_t *ng = reinterpret_cast<uint32_t *>(outs[9].p);
    k_split<<<8, kThreads>>>(reinterpret_cast<int32_t *>(d_rows), m, n, 0, 1, as32(0), as32(1), as32(2),
                             reinterpret_cast<int64_t *>(outs[3].p), word, err);
    std::vector<int32_t> src(m);
    for (int64_t e = 0; e < m; ++e) src[e] = rows[e].x;
    int32_t *d_src;
    cudaMalloc((void **)&d_src, 4 * m);
    cudaMemcpy(d_src, src.data(), 4 * m, cudaMemcpyHostToDevice);
    k_filter<<<8, kThreads>>>(d_src, fixed_adj, fixed_lab, m, nword, as64(4), err);
    k_regions<<<8, kThreads>>>(d_rows, m, 0, fixed_off, as64(5), err);
    k_hash<<<8, kThreads>>>(d_src, fixed_adj, fixed_lab, m, nbkt, reinterpret_cast<int4 *>(outs[6].p), word, err);
    k_group_lists<<<8, kThreads>>>(fixed_off, fixed_adj, fixed_lab, d_vlab, n, m, C, as32(7), as32(8), ng, as32(10),
                                   word + 2, err);
    k_group_hubs<<<2, 1024>>>(fixed_off, fixed_adj, fixed_lab, d_vlab, C, as32(11), as32(8), ng, d_hub,
                              reinterpret_cast<uint32_t *>(d_hub + 1), err);
    if (cudaDeviceSynchronize() != cudaSuccess) return 2;
    cudaFree(d_src);
    for (Out &o : outs) {
      std::vector<unsigned char> h(o.bytes);
      cudaMemcpy(h.data(), o.p, o.bytes, cudaMemcpyDeviceToHost);
      bool changed = false;
      for (unsigned char c : h) changed |= c != h[0];
      const unsigned char fill = &o == &outs[6] ? 0xff : &o == &outs[4] || &o == &outs[5] ? 0 : 0x5a;
      changed |= h[0] != fill;
      if (changed != (failed == 0)) {
        std::printf("%s: %s with the word %s\n", o.name, changed ? "written" : "not written", failed ? "set" : "clear");
        ++bad;
      }
    }
  }
  std::puts(bad ? "bad" : "ok");
  return bad != 0;
}
"""


def test_nothing_is_indexed_by_rows_of_a_failed_sort(tmp_path):
    from paper_2507_04130_gb300 import _build

    src = tmp_path / "harness.cu"
    src.write_text(_HARNESS)
    exe = str(tmp_path / "harness")
    cmd = [_build._nvcc(), *_build.ARCH, "-O1", "-std=c++17", f"-I{_build.INCLUDE}", f"-I{_build.CSRC}", str(src),
           *[os.path.join(_build.CSRC, f) for f in ("hm_sort.cu", "hm_api.cpp")], "-o", exe]
    made = subprocess.run(cmd, capture_output=True, text=True)
    assert made.returncode == 0, made.stderr
    ran = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert ran.returncode == 0 and ran.stdout.strip() == "ok", ran.stdout + ran.stderr
