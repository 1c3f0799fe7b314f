"""Device memory of a context: what it takes where rows of Y_(n) are wide and slices long (the partial rows
of cut slices, P_n floats for each piece; measured in a process of its own, from cudaMemGetInfo), and what
runs without the part of it that is optional."""
import subprocess
import sys

import pytest

from paper_2010_10638_gb300 import synth
from tests.conftest import ROOT
from tests.gpu_util import lib

pytestmark = pytest.mark.gpu

CODE = """
import torch
from paper_2010_10638_gb300 import tucker as T
T.load()
g = torch.Generator(device="cuda").manual_seed(1)
dims, ranks, nnz = (100, 300, 300, 2000), (2, 64, 64, 16), 2_500_000
coords = torch.stack([torch.randint(0, d, (nnz,), generator=g, device="cuda", dtype=torch.int32) for d in dims])
vals = torch.randn(nnz, generator=g, device="cuda")
T.tucker_lib_setup()
torch.cuda.synchronize()
before = torch.cuda.mem_get_info()[0]
ctx = T.tucker_init(dims, coords, vals, ranks, seed=2)
torch.cuda.synchronize()
after = torch.cuda.mem_get_info()[0]
Y = T.ttmc_mode(ctx, 0)
rows = torch.zeros_like(Y)  # the same in FP64, from FP32 factors, one slice
U = [T.tucker_get_factor(ctx, m).float().double() for m in range(4)]
sel = coords[0] == 7
c, v = coords[:, sel].long(), vals[sel].double()
left = (U[1][c[1]].unsqueeze(2) * U[2][c[2]].unsqueeze(1)).reshape(c.shape[1], -1)
ref = ((left * v[:, None]).T @ U[3][c[3]]).reshape(-1)
print(before - after, float((Y[7].double() - ref).norm() / ref.norm()))
"""


def test_wide_rows_and_long_slices():
    """100 slices of 25,000 nonzeros and P_1 = 65,536.  Partial rows of pieces of 2,048 nonzeros take 0.35 GB,
    the copies and their sort 0.4, the core's partials 0.32, the rest below 0.1; twice the sum leaves room
    for what the allocator rounds up.  In pieces of 256 nonzeros the partial rows alone take 2.6 GB."""
    lib()
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    used, err = r.stdout.split()
    assert float(err) <= 1e-5
    assert int(used) <= 2.34e9, used


def test_the_optional_workspace_is_allocated_last(monkeypatch):
    """Of the allocations of tucker_init only the last, the workspace of the QRP's Gram form, may fail
    without the call failing: it takes no memory that another one needs.  Without it a sweep is that of
    the cluster form, bit for bit."""
    T = lib()
    w = synth.make("tiny-100^3")
    args = w.workload.dims, w.coords, w.vals, w.workload.ranks, w.U0
    worked = []
    for k in range(1, 200):
        monkeypatch.setenv("TUCKER_FAIL_ALLOC_AT", str(k))
        try:
            ctx = T.tucker_init(*args)
        except T.TuckerError as e:
            assert e.name == "TUCKER_ENOMEM"
            worked.append(False)
        else:
            if not any(worked):
                fit = T.hooi_iter(ctx)
            worked.append(True)
            T.tucker_free(ctx)
    first = worked.index(True)
    assert 20 < first and all(worked[first:])
    monkeypatch.delenv("TUCKER_FAIL_ALLOC_AT")
    monkeypatch.setenv("TUCKER_QRP_FORM", "cluster")
    assert T.hooi_iter(T.tucker_init(*args)) == fit
