"""Buffers aligned to no more than their element types: bakron_prepare's wide loads
sit on 32-byte boundaries inside whatever it is given.
"""
import ctypes
import subprocess

import pytest
import torch

import workloads as WL
from paper_2608_06291_gb300 import buildlib

CSRC = buildlib.CSRC

PLACES = r"""
#include "common.cuh"
#include <cstdio>
#include <algorithm>
#include <utility>
#include <vector>
using namespace bakron;
int main() {
  for (int m : {1, 128, 129, 700}) for (int n : {1, 64, 385, 1000}) for (int o = 0; o < 64; o += 4) {
    FactorLayout fl(m, n);
    PrepareLayout pl(m, n);
    char *f = (char*)4096 + o, *w = (char*)(size_t(1) << 40) + 4 * (o / 4 * 7 % 16);
    PrepareScratch s(fl, pl, f, w);
    const size_t a = fl.np, b = fl.mp, small = 64 * 8 + 8 + 16 + 5 * 4;
    typedef std::pair<char*, char*> R;
    std::vector<R> rf = {R(s.CA, s.CA + a * a * 8), R(s.CB, s.CB + b * b * 8),
                         R(s.smallA, s.smallA + a * small), R(s.smallB, s.smallB + b * small)};
    std::vector<R> rw = {R(w, w + 256), R(s.XA, s.XA + a * a * 8), R(s.XB, s.XB + b * b * 8)};
    auto check = [&](std::vector<R>& r, char* base, size_t bytes) {
      for (auto& x : r) {
        if (x.first < base || x.second > base + bytes) return false;
        if (x.first != w && (size_t)x.first % 32) return false;
      }
      std::sort(r.begin(), r.end());
      for (size_t i = 1; i < r.size(); ++i)
        if (r[i].first < r[i - 1].second) return false;
      return true;
    };
    if (!check(rf, f, fl.bytes) || !check(rw, w, pl.bytes)) {
      std::printf("m %d n %d offset %d\n", m, n, o);
      return 1;
    }
    // the last step writes the leaf blocks of both sides, then nothing of C is read:
    // C may only reach over the planes into rB
    if (s.CA + a * a * 8 > f + fl.off_rA) return 1;
  }
  return 0;
}
"""


def test_scratch_is_aligned_inside_the_buffers(tmp_path):
    src = tmp_path / "places.cu"
    src.write_text(PLACES)
    exe = tmp_path / "places"
    subprocess.run([buildlib.nvcc(), *buildlib.ARCH, "-std=c++17", "-I", CSRC, "-I", buildlib.INCLUDE,
                    str(src), "-o", str(exe)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("off_f,off_w", [(16, 16), (0, 8), (4, 0), (20, 12)])
def test_prepare_with_offset_buffers(off_f, off_w):
    import paper_2608_06291_gb300 as P
    P.build()
    m, n = 200, 300
    _, A, B = WL.small_problem(m, n, 3)
    A, B = A.cuda(), B.cuda()
    want = P.bakron_get_factors(P.bakron_prepare(A, B, 0.01))
    f = P.Factors(m, n)
    size = f.buf.numel()
    f.buf = torch.full((size + 64,), 0xff, dtype=torch.uint8, device="cuda")[off_f:off_f + size]
    ws = torch.full((P.workspace_bytes(m, n) + 64,), 0xff, dtype=torch.uint8, device="cuda")[off_w:off_w - 64]
    assert f.buf.data_ptr() % 32 == off_f and ws.data_ptr() % 32 == off_w
    vp = ctypes.c_void_p
    rc = P.lib().bakron_prepare(vp(A.data_ptr()), vp(B.data_ptr()), m, n, 0.01, vp(f.buf.data_ptr()),
                                vp(ws.data_ptr()), ws.numel(), vp(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    for got, ref in zip(P.bakron_get_factors(f), want):
        assert torch.equal(got, ref)
