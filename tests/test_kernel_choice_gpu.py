"""The kernels that a setting names are the ones that run, and the autotuners
time what the steps they tune for would run (GPU required)."""
import re

import numpy as np
import pytest

from test_ensemble_gpu import make, same

pytestmark = pytest.mark.gpu

COMMON = dict(G=1.5, eta_p=0.1, tau_p=20.0, L2=50.0, kappa=0.01, phase=1)


@pytest.fixture(scope="module", autouse=True)
def profiler():
    """The first session of a process records nothing: it starts the tracing."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]):
        torch.zeros(1, device="cuda")
        torch.cuda.synchronize()


def launched(call):
    """{kernel name: launches} of a call."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    names = {}
    for e in prof.key_averages():
        m = re.search(r"\b(k_[a-z0-9_]+)", e.key)
        if m:
            names[m.group(1)] = names.get(m.group(1), 0) + e.count
    return names


@pytest.mark.parametrize("variant", ["walls", "periodic", "one_component", "fp16", "bf16_walls", "mrt", "chol"])
def test_post_mode_set_is_the_pass_that_runs(variant):
    """Below the size up to which the default takes the runs, post mode 2 marches
    columns once it is set, mode 1 takes the runs, and both leave the default's bits."""
    box = dict(COMMON, lattice=1, nx=64, ny=16, nz=11, ncomp=2, walls=1, u_wall=0.03)
    box.update({"periodic": dict(walls=0, u_wall=0.0, fext=(1e-5, -1e-5, 0.0)),
                "one_component": dict(ncomp=1, G=0.0, phase=0), "fp16": dict(walls=0, u_wall=0.0, precision=1),
                "bf16_walls": dict(precision=2)}.get(variant, {}))
    lats = {}
    for config, kernel in ((None, "k_post"), ((0, 1), "k_post"), ((0, 2), "k_post_zm")):
        L = lats[config] = make(box, seed=17)
        L.set_collision(int(variant == "mrt"))
        L.set_conformation_update(int(variant == "chol"))
        if config:
            L.set_kernel_config(*config)
        L.set_step_graph(0)
        L.step(1)
        names = launched(lambda: L.step(4))
        assert [k for k in names if k.startswith("k_post")] == [kernel], (config, names)
    assert same(lats[None], lats[(0, 1)]) and same(lats[None], lats[(0, 2)])


def test_autotune_keeps_the_many_step_launch():
    """On a small D2Q9 lattice tile 0 is timed with the launches of many steps
    that it admits, which no other tile comes near (1.6 against 3.5 us a step)."""
    L = make(dict(COMMON, lattice=0, nx=64, ny=32, ncomp=1, walls=1, u_wall=0.03, G=0.0), seed=5)
    for steps in (50, 1):
        times = L.autotune(steps=steps)
        assert L.kernel_config()[0] == 0, times
    assert "k_small" in launched(lambda: L.step(20))


def test_autotune_times_the_step_graph():
    """Pairs that admit the slab graph are timed with it: 128 x 32 x 112 takes 4
    slabs, so tiles 0-2 with the marching pass launch it four times a step."""
    L = make(dict(COMMON, lattice=1, nx=128, ny=32, nz=112, ncomp=2, walls=1, u_wall=0.03), seed=6)
    assert L.step_graph[0] == 4
    names = launched(lambda: L.autotune(steps=8))
    # eager, each of 6 tiles (and the fused pair) would launch it 16 times: 112
    assert names["k_post_zm"] >= 3 * 16 * 4, names


def test_ensemble_form_set_is_the_form_that_runs():
    """Members of 2^14 nodes and more step in branches until batched launches are
    set, which then run, also with tile 0 and the automatic segment and groups."""
    from paper_1406_2686_gb300 import vefd
    sizes = [(64, 32, 16), (32, 32, 33), (64, 16, 20)]
    boxes = [dict(COMMON, lattice=1, nx=x, ny=y, nz=z, ncomp=2, walls=1, u_wall=0.03) for x, y, z in sizes]
    E = vefd.Ensemble([make(b, seed=30 + k) for k, b in enumerate(boxes)])
    for ask, batched in ((None, False), (True, True), (False, False)):
        if ask is not None:
            E.set_batched(ask)
        E.step(9, chunk=4)
        assert E.batched == batched and E.config == (0 if ask is False else 1, 0)
    E.set_config(True, 0)
    E.step(4, chunk=4)
    assert E.batched
    times = E.autotune(steps=8, chunk=4)
    assert all(t > 0 for t in times), times  # every configuration: the members allow batched launches
    best = int(np.argmin(times))
    assert E.config[0] == int(best > 0)
    E.step(8, chunk=4)
    assert E.batched == (best > 0)
    E.close()
