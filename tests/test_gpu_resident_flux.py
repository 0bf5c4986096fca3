"""The resident kernels of the flux form (patches of the mesh in shared memory)
against the launches per step, which carry calls and checkpoint intervals of
fewer than 16 steps: the same bits, in two and three dimensions, with and
without layers, ragged shot counts, and as the recompute of J^T w; a wait that
runs out raises."""
import numpy as np
import pytest

from workloads import configs

pytestmark = pytest.mark.gpu


@pytest.fixture()
def mg(cuda_device):
    import paper_1707_04605_gb300 as m

    return m


def cu(x, t=None):
    import torch

    return torch.as_tensor(np.ascontiguousarray(x), dtype=t or torch.float64, device="cuda")


CASES = [
    (configs.asteroid_2d, dict(n_refine=1, S=1, nt=41)),      # one patch per 32 rows
    (configs.asteroid_2d, dict(n_refine=1, S=10, nt=17)),     # columns beyond the shots
    (configs.asteroid_2d, dict(n_refine=2, S=37, nt=40)),     # a ragged last column group
    (configs.asteroid_2d, dict(n_refine=1, S=130, nt=20)),    # two groups of 32 lanes
    (configs.asteroid_2d, dict(n_refine=3, S=12, nt=24)),     # patches that fill an SM
    (configs.ellipsoid_3d, dict(n_refine=0, S=5, nt=33)),
    (configs.tiny_3d, dict(nt=20)),
    (configs.tiny_2d, dict(nt=30)),
]


def setup(mg, make, kw, layer):
    w = make(**kw)
    m = w.mesh
    mesh = mg.mesh_from_workload(w)
    rng = np.random.default_rng(3)
    xi = cu(rng.uniform(0.0, 2.0, m.n_cells[-1])) if layer else None
    zeta = cu(rng.uniform(0.0, 2.0, (m.n_cells[-1], m.coords.shape[1]))) if layer else None
    eps = cu(w.eps)
    dt = 0.4 * mg.cfl_dt(mesh, eps)
    return w, mesh, eps, dt, cu(w.wavelet(dt)), xi, zeta


@pytest.mark.parametrize("layer", [False, True])
@pytest.mark.parametrize("make,kw", CASES)
def test_resident_flux_carries_the_bits_of_the_steps(mg, make, kw, layer):
    import torch

    w, mesh, eps, dt, wav, xi, zeta = setup(mg, make, kw, layer)
    n0 = mesh.launch_count()
    y = mg.forward_pml(mesh, eps, w.shots, wav, dt, xi, zeta)
    assert mesh.launch_count() - n0 < 2 * w.nt
    few = mg.forward_pml(mesh, eps, w.shots, wav[:15].contiguous(), dt, xi, zeta)
    assert few.abs().max() > 0 and torch.equal(y[:, :15], few)
    W = cu(np.random.default_rng(5).standard_normal(y.shape), torch.float32)
    steps = mg.jacobian_T_apply_pml(mesh, 0, eps, w.shots, wav, dt, W, xi, zeta, ckpt_every=8)
    for ck in (16, w.nt):   # recomputed segments (the last one shorter), kept states
        g = mg.jacobian_T_apply_pml(mesh, 0, eps, w.shots, wav, dt, W, xi, zeta, ckpt_every=ck)
        assert torch.equal(g, steps)


def test_a_flux_wait_that_runs_out_raises(mg):
    w, mesh, eps, dt, wav, xi, zeta = setup(mg, configs.asteroid_2d,
                                            dict(n_refine=2, S=16, nt=64), False)
    y = mg.forward_pml(mesh, eps, w.shots, wav, dt)
    mesh.set_persistent(wait_cycles=1000)        # below one exchange of border rows
    with pytest.raises(Exception, match="(?i)time|wait"):
        mg.forward_pml(mesh, eps, w.shots, wav, dt)
    mesh.set_persistent()
    assert mg.forward_pml(mesh, eps, w.shots, wav, dt).equal(y)


def test_a_large_call_does_not_wait_for_other_streams(mg):
    """Work buffers above what a handle keeps (2 GB) are allocated and freed in the
    order of the call's own stream (launches per step: they need no SM to
    themselves)."""
    import torch

    w = configs.asteroid_2d(n_refine=4, S=256, nt=6)
    m = mg.mesh_from_workload(w)
    eps = cu(w.eps)
    dt = 0.5 * mg.cfl_dt(m, eps)
    s = cu(w.wavelet(dt))
    v = cu(np.ones(w.mesh.n_cells[0]))
    run = lambda: mg.jacobian_apply_pml(m, 0, eps, w.shots, s, dt, v)
    ref = run()
    n, cells = w.mesh.coords.shape[0], len(w.mesh.cells)
    assert 4 * 256 * (2 * n + 4 * cells) > 2 << 30   # p, dp, q and dq
    side, done = torch.cuda.Stream(), torch.cuda.Event()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(3_000_000_000)             # more than a second
        done.record()
    jv = run()
    assert not done.query()
    assert torch.equal(jv, ref)
    torch.cuda.synchronize()


def test_trim_and_info_beside_a_call_of_another_thread(mg):
    """Flux calls of several threads on one handle (each with its own stream and
    work buffers) while the handle's kept buffers are counted and given back."""
    import threading

    import torch

    w = configs.asteroid_2d(n_refine=1, S=10, nt=12)
    m = mg.mesh_from_workload(w)
    eps = cu(w.eps)
    dt = 0.5 * mg.cfl_dt(m, eps)
    s = cu(w.wavelet(dt))
    ref = mg.forward_pml(m, eps, w.shots, s, dt, allow_cfl=True)
    torch.cuda.synchronize()
    wrong, left = [], [3]

    def calls():
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(40):
                    if not torch.equal(mg.forward_pml(m, eps, w.shots, s, dt, allow_cfl=True), ref):
                        wrong.append(1)
        except Exception as e:
            wrong.append(e)
        left[0] -= 1

    threads = [threading.Thread(target=calls) for _ in range(left[0])]
    for t in threads:
        t.start()
    while left[0] > 0:
        assert m.info()["device_bytes"] > 0
        m.trim()
    for t in threads:
        t.join()
    assert not wrong
