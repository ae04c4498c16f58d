"""The source gradient on tall boxes with few antenna columns, where 2, 4 or 8
CTAs share the planes of 32 columns (from 65, 129 and 257 planes on), against the
oracle's adjoint; 64 planes take one CTA."""
import numpy as np
import pytest
import torch

import oracle
from paper_2102_12978_gb300 import fdtd
from paper_2102_12978_gb300 import workloads as W
from tests.cases import oracle_grid, oracle_source, rel_l2
from tests.gpu_cases import gpu_grid, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [("f64", 1e-10), ("f32", 1e-3)])
@pytest.mark.parametrize("nx,ny,nz,r,thick", [(28, 26, 64, 7.0, 1.0), (28, 26, 65, 7.0, 1.0), (26, 30, 131, 6.0, 3.0),
                                              (24, 25, 257, 6.0, 1.0), (41, 37, 300, 12.0, 2.0)])
def test_gradient_matches_oracle(nx, ny, nz, r, thick, precision, tol):
    w = W.small(nx=nx, ny=ny, nz=nz, npml=4, r_center=r, thickness=thick, steps=7, ramp=0.1, theta_deg=25.0)
    amp, ph = W.random_weights(w.nx, w.ny, seed=3)
    g = gpu_grid(w, precision, fluence=False, w_amp=amp, w_phase=ph)
    rng = W.rng(9)
    probes = rng.choice(nx * ny * nz, size=400, replace=False)
    dlde = rng.standard_normal((4, probes.size))
    adj = fdtd.Adjoint(g, fdtd.EY, probes)
    adj.reset(w.steps)
    adj.step(4, torch.tensor(dlde, device=g.device))
    adj.step(w.steps - 4)
    ga, gp = (host(t) for t in adj.gradient())
    og = oracle_grid(w)
    src = oracle_source(w, w_amp=amp, w_phase=ph)
    ao = oracle.State(og, fluence=False)
    gao, gpo = np.zeros((ny, nx)), np.zeros((ny, nx))
    for q, n in enumerate(reversed(range(w.steps))):
        if q < 4:
            np.add.at(ao.e[1].reshape(-1), probes, dlde[q])
        oracle.adjoint_step(og, src, ao, n, gao, gpo)
    assert np.abs(gao).max() > 0
    assert rel_l2(ga, gao) <= tol, rel_l2(ga, gao)
    assert rel_l2(gp, gpo) <= tol, rel_l2(gp, gpo)
    again = fdtd.Adjoint(g, fdtd.EY, probes)     # the sums are taken in a fixed order
    again.reset(w.steps)
    again.step(4, torch.tensor(dlde, device=g.device))
    again.step(w.steps - 4)
    for x, y in zip(adj.gradient(), again.gradient()):
        assert torch.equal(x, y)
