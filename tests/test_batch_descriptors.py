"""What solve_batch hands to the library: the descriptor array's fields, in host
memory whatever PyTorch's default device (a stand-in for the library reads
them; no GPU)."""
import ctypes

import pytest
import torch

M = pytest.importorskip("paper_2607_23354_gb300")

# 1 to 256 problems are formed as lists, more as tensors


class _Library:
    def mag_solve_batch(self, h, desc, count, points, w, mags, status, info):
        self.rows = [(d.point_offset, d.w_offset, d.n, d.m, d.t) for d in desc[:count]]
        ctypes.memset(status, 0, 4 * count)
        return M.MAG_OK


def _solve_batch(clouds, ts):
    c = M.Context.__new__(M.Context)
    c.device, c._lib, c._h = torch.device("cpu"), _Library(), None
    ws, mags, sts = c.solve_batch(clouds, ts)
    return c._lib.rows, ws, mags, sts


@pytest.mark.parametrize("sizes,ts", [([(3, 2)], [0.5]), ([(5, 4)], [1.0, 2.0]), ([(7, 1), (2, 9), (300, 16)], [1e-3, 7.0, 1e5]),
                                      ([(2 + i, 3) for i in range(128)], [2.0, 3.0]),
                                      ([(2 + i, 3) for i in range(257)], [2.0]), ([(2 + i, 3) for i in range(700)], [2.0, 3.0])])
@pytest.mark.parametrize("default", ["cpu", "meta"])
def test_descriptors(sizes, ts, default):
    clouds = [torch.zeros(n, m, dtype=torch.float64) for n, m in sizes]
    with torch.device(default):
        rows, ws, mags, sts = _solve_batch(clouds, ts)
    want, p, w = [], 0, 0
    for n, m in sizes:
        for t in ts:
            want.append((p, w, n, m, t))
            w += n
        p += n * m
    assert rows == want
    assert [len(v) for v in ws] == [r[2] for r in want]
    assert mags.shape == sts.shape == (len(sizes), len(ts)) and not sts.any()
