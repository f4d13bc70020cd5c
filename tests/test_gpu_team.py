"""Teams of threads per zone (csrc/coop.cuh): how many threads share a zone
is chosen from the number of zones and the network, and must not change a
bit.  The same zones are burned (and differentiated) among fewer and more
zones, on both sides of every line of the rule."""
import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu


def _setup(name, Z, t_end=None):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2312_02836_gb300 as nb
    net, z, s = gen.problem(name, Z)
    t = {k: torch.from_numpy(v).cuda() for k, v in z.items()}
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    return nb, torch, nb.Network(net), t, (t_end or s["t_end"], s["rtol"], s["atol"]), sm


def _first(t, n):
    return [t[k][:n].contiguous() for k in ("Y", "T9", "rho")]


def _same(torch, a, b, n):
    for x, y in zip(a, b):
        assert torch.equal(x[:n], y[:n])


@pytest.mark.parametrize("name,t_end", [("net48", 1e-4), ("chain13_heat", 1e-5)])
@pytest.mark.parametrize("wpz", [0, 2, 4])
def test_threads_per_zone_keep_the_bits(name, t_end, wpz):
    nb, torch, net, t, tol, sm = _setup(name, 3000, t_end)
    full = nb.burn(net, *_first(t, 3000), *tol, kernel="coop", warps_per_zone=wpz)
    for Z in (1, 3, 6 * sm, 6 * sm + 1, 16 * sm, 16 * sm + 1):
        out = nb.burn(net, *_first(t, Z), *tol, kernel="coop", warps_per_zone=wpz)
        _same(torch, out, full, Z)
    out = nb.burn(net, *_first(t, 100), *tol, kernel="coop", warps_per_zone=wpz, ws_in_shared=0)
    _same(torch, out, full, 100)


def test_threads_per_zone_keep_the_bits_of_a_large_network():
    nb, torch, net, t, tol, sm = _setup("net128_heat", 40, 1e-7)
    for wpz in (0, 2, 4):
        full = nb.burn(net, *_first(t, 40), *tol, kernel="coop", warps_per_zone=wpz)
        out = nb.burn(net, *_first(t, 7), *tol, kernel="coop", warps_per_zone=wpz, ws_in_shared=0)
        _same(torch, out, full, 7)


@pytest.mark.parametrize("name,t_end,K", [("net48_adjoint", 1e-4, 3), ("chain13_heat", 1e-5, 1),
                                          ("net128_heat", 1e-8, 2)])
def test_adjoint_threads_per_zone_keep_the_bits(name, t_end, K):
    big = 1500 if name != "net128_heat" else 24
    nb, torch, net, t, tol, sm = _setup(name, big, t_end)
    rng = np.random.default_rng(3)
    gY = torch.from_numpy(rng.normal(size=(K, big, net.N))).cuda()
    gE = torch.from_numpy(rng.normal(size=(K, big))).cuda()

    def grads(Z, **opt):
        tape = nb.Tape(net, Z, 600)
        nb.burn(net, *_first(t, Z), *tol, kernel="coop", tape=tape)
        return nb.adjoint(net, tape, gY[:, :Z].contiguous(), gE[:, :Z].contiguous(), **opt)

    full = grads(big)
    sizes = (1, 8 * sm, 8 * sm + 1) if name != "net128_heat" else (1, 9)
    for Z in sizes:
        for x, y in zip(grads(Z), full):
            assert torch.equal(x, y[:, :Z])
    for x, y in zip(grads(9, kernel="coop", ws_in_shared=0), full):
        assert torch.equal(x, y[:, :9])
