"""J^T w of the flux form with shot counts whose float4 groups are neither a
power of two nor a multiple of 32: the node adjoint's sum over the shots is
taken over whole groups, so the gradient matches the FP64 oracle."""
import numpy as np
import pytest

from helpers import JAC_TOL, rel_l2
from oracle import mixed, wave
from workloads import configs, shots as shots_mod

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [10, 23, 140])
def test_ragged_shot_counts_match_oracle(cuda_device, S):
    import torch

    import paper_1707_04605_gb300 as mg

    w = configs.tiny_2d(nt=40)
    m = w.mesh
    rng = np.random.default_rng(S)
    n = m.coords.shape[0]
    sh = shots_mod.Shots(rng.integers(0, n, S).astype(np.int32), np.arange(S + 1, dtype=np.int64),
                         rng.integers(0, n, S).astype(np.int32))
    dt = 0.5 * wave.Problem(m.coords, m.cells, m.bnd, w.eps, "neumann").cfl_dt()
    s = w.wavelet(dt)
    xi, zeta = mixed.square_layer(m.coords, m.cells, 0.7, 1.0, 5.0)
    W = rng.standard_normal((S, w.nt)).astype(np.float32)
    mesh = mg.mesh_from_workload(w)
    t = lambda x, d=torch.float64: torch.as_tensor(np.ascontiguousarray(x), dtype=d, device="cuda")
    g = mg.jacobian_T_apply_pml(mesh, 1, t(w.eps), sh, t(s), dt, t(W, torch.float32), t(xi),
                                t(zeta), ckpt_every=16).cpu().numpy()
    ref = mixed.adjoint_eps(m.coords, m.cells, w.eps, dt, s, sh.src, sh.rec_ptr, sh.rec,
                            W.astype(np.float64), xi=xi, zeta=zeta)
    assert rel_l2(g, wave.restrict(ref, m.ancestor(1), m.n_cells[1])) < JAC_TOL
