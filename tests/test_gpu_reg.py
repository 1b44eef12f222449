"""Fused momentum-space kernels below N_x = 16: the weak-coupling preconditioner, whose M1 terms run
on them, against the oracle at every extent (ragged N_tau), and a batch of one extent whose N_tau is
no multiple of the slices per tile.  Tolerances as for the other weak-coupling parity tests: FP64
1e-11, FP32 1e-4 (d + 1 exact inverses of O(N_tau + 3N) rounding steps each)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1008_3647_gb300.inputs import field_and_source

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ufg():
    from paper_1008_3647_gb300 import ufg as u
    u.load()
    return u


@pytest.mark.parametrize("dtype,tol", [(torch.float64, 1e-11), (torch.float32, 1e-4)])
@pytest.mark.parametrize("transpose", [False, True])
@pytest.mark.parametrize("nx,ntau", [(4, 3), (4, 37), (6, 11), (8, 5), (10, 7), (12, 9)])
def test_wce_parity_small_extents(ufg, nx, ntau, transpose, dtype, tol):
    sigma, r = field_and_source(nx, ntau, 60 + nx + ntau)
    lat = ufg.Lattice(nx, ntau)
    field = ufg.Field(lat, torch.from_numpy(sigma).cuda())
    solver = ufg.Solver(lat)
    solver.ufg_set_preconditioner("wce", order=2, euler="euler23")
    rd = torch.from_numpy(r).to("cuda", dtype)
    z = solver.ufg_apply_preconditioner(field, rd, transpose=transpose).double().cpu().numpy()
    fn = O.wce_apply_T if transpose else O.wce_apply
    ref = fn(O.Lattice(nx, ntau), sigma, rd.double().cpu().numpy(), 2, "euler23")
    assert float(np.abs(z - ref).max() / np.abs(ref).max()) < tol


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("shapes", [[(6, 13), (6, 41), (6, 8)], [(10, 9), (12, 7), (4, 21), (8, 11)]])
def test_batches_with_ragged_tiles(ufg, shapes, mixed):
    probs = []
    for i, (nx, nt) in enumerate(shapes):
        sg, b = field_and_source(nx, nt, 70 + i)
        probs.append({"nx": nx, "ntau": nt, "sigma": torch.from_numpy(sg).cuda(),
                      "b": torch.from_numpy(b).cuda(),
                      "x": torch.zeros(b.shape, dtype=torch.float64, device="cuda")})
    stats = ufg.ufg_solve_batch(probs, "wce", dict(order=2, euler="euler23"), tol=1e-10,
                                precision=ufg.UFG_MIXED if mixed else ufg.UFG_FP64)
    for (nx, nt), pr, st in zip(shapes, probs, stats):
        assert st["status"] == ufg.UFG_OK, st
        b = pr["b"].cpu().numpy()
        r = b - O.apply_Q(O.Lattice(nx, nt), pr["sigma"].cpu().numpy(), pr["x"].cpu().numpy())
        assert np.linalg.norm(r) <= 1e-10 * np.linalg.norm(b)
    ufg.ufg_batch_cache_clear()
