"""The reset's risk test at its line: quotients of D_Q and D_M that round to tau and to its neighbours, and operands and limits for which a
product says nothing (zeros, subnormal and huge values, infinities, NaN, limits that are zero, negative, subnormal or infinite). The elements
that are reset are those whose binary32 quotient is at least tau."""

import numpy as np
import pytest
import torch

from paper_2510_27527_b200 import binding as b

pytestmark = pytest.mark.gpu

TAUS = [6.0, 1.0, 0.3, float(np.nextafter(np.float32(2), np.float32(0))), 3e38, 1e-38, 1e-42, 2.0**-100, 2.0**-99, 0.0, -1.0, float("inf")]


@pytest.mark.parametrize("tau", TAUS)
@pytest.mark.parametrize("cols", [128, 127, 1000])
def test_reset_elements_are_those_at_or_above_the_line(tau, cols):
    rng = np.random.RandomState(3)
    rows = 64
    t = np.float32(tau)
    with np.errstate(all="ignore"):
        dm = (rng.rand(rows, cols).astype(np.float32) + np.float32(0.01)) * np.float32(2.0) ** rng.randint(-20, 20, (rows, cols)).astype(np.float32)
        dq = dm * t  # within an ulp of the line; then up to 12 ulps to either side of it
        for _ in range(12):
            step = rng.randint(-1, 2, dq.shape)
            dq = np.where(step > 0, np.nextafter(dq, np.float32(np.inf)), np.where(step < 0, np.nextafter(dq, np.float32(-np.inf)), dq)).astype(np.float32)
        far = rng.rand(rows, cols)
        dq = np.where(far < 0.2, dq * np.float32(1.5), np.where(far < 0.4, dq * np.float32(0.5), dq)).astype(np.float32)
        odd = np.array([0.0, -0.0, 1e-45, 1e-38, 3e38, np.inf, np.nan, 1.0, 2.0**-110, 2.0**110], dtype=np.float32)
        pick = rng.rand(rows, cols) < 0.1
        dm = np.where(pick, odd[rng.randint(0, len(odd), dm.shape)], dm)
        dq = np.where(pick | (rng.rand(rows, cols) < 0.05), odd[rng.randint(0, len(odd), dq.shape)], dq)
        want = (dq / dm >= t) & ~((dq == 0) & (t > 0))
    w0 = torch.from_numpy((rng.randn(rows, cols) + 0.01).astype(np.float32)).cuda()
    # Q(W): what a reset of every element leaves
    full = w0.clone()
    ones = torch.ones_like(w0)
    b.nvfp4_osci_suppress(full, b.OsciState(w0.clone(), ones, 2 * ones), 1.0, b.GS_TENSOR)
    w, n = w0.clone(), torch.zeros(1, dtype=torch.int64, device="cuda")
    b.nvfp4_osci_suppress(w, b.OsciState(w0.clone(), torch.from_numpy(dm).cuda(), torch.from_numpy(dq).cuda()), float(t), b.GS_TENSOR, n_reset=n)
    assert int(n) == int(want.sum())
    assert torch.equal(w, torch.where(torch.from_numpy(want).cuda(), full, w0))
