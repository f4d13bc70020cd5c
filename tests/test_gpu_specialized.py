"""The network-specialised kernel (CUDA generated per network, compiled at
run time) against the generic kernel.  Both perform the same floating-point
operations in the same order, so every output must be equal bit for bit,
for every storage variant and every option that changes the integration
(per-zone multipliers, per-zone end times, the adjoint tape).  Parity with
the oracle is checked by the parity tests, which run both kernels."""
import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu


def _setup(name, Z):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2312_02836_gb300 as nb
    net, z, s = gen.problem(name, Z)
    dev = torch.device("cuda")
    t = {k: torch.from_numpy(v).to(dev) for k, v in z.items()}
    return nb, torch, net, z, s, t


def _equal(a, b):
    import torch
    for x, y in zip(a, b):
        assert torch.equal(x, y)


CASES = [("chain13", 2048), ("chain13_literal", 1024), ("chain13_heat", 2048),
         ("chain13_heat_ap", 1024), ("chain13_heat_scr", 1024), ("chain13_heat_tab", 1024)]


@pytest.mark.parametrize("variant", [1, 2, 3])
@pytest.mark.parametrize("name,Z", CASES)
def test_specialized_equals_generic_bitwise(name, Z, variant):
    nb, torch, net, z, s, t = _setup(name, Z)
    nc = nb.Network(net)
    args = (nc, t["Y"], t["T9"], t["rho"], s["t_end"], s["rtol"], s["atol"])
    zk = dict(zeta=t["zeta"]) if "zeta" in t else {}
    ref = nb.burn(*args, specialize="generic", **zk)
    assert nc.info()["last_specialized"] == 0
    out = nb.burn(*args, specialize=variant, **zk)
    torch.cuda.synchronize()
    assert nc.info()["last_specialized"] == variant
    assert int((out.status == 0).sum()) == Z
    _equal(out, ref)
    # other launch shapes of the specialised kernel: the same bits
    for tpb, bps in ((64, 1), (128, 2), (256, 1)):
        again = nb.burn(*args, specialize=variant, threads_per_block=tpb,
                        blocks_per_sm=bps, schedule="fifo", **zk)
        torch.cuda.synchronize()
        _equal(again, ref)


def test_automatic_choice():
    nb, torch, net, z, s, t = _setup("chain13_heat", 512)
    nc = nb.Network(net)
    info = nc.info()
    assert info["specialize_auto"] == 1
    nb.burn(nc, t["Y"], t["T9"], t["rho"], s["t_end"], s["rtol"], s["atol"])
    torch.cuda.synchronize()
    assert nc.info()["last_specialized"] in (1, 2, 3)
    nb.burn(nc, t["Y"], t["T9"], t["rho"], s["t_end"], s["rtol"], s["atol"],
            kernel="plain")
    assert nc.info()["last_specialized"] == 0
    # a network too large for straight-line code stays on the generic kernel
    big = nb.Network(gen.network("net128_heat"))
    assert big.info()["specialize_auto"] == 0
    log = nc.specialize(3)
    assert "error" not in log.lower()


def test_specialized_options_and_tape_bitwise():
    # per-zone rate multipliers, per-zone end times and the recorded tape:
    # the adjoint of the two tapes must agree to the bit as well
    name, Z = "chain13_heat", 1024
    nb, torch, net, z, s, t = _setup(name, Z)
    nc = nb.Network(net)
    rng = np.random.default_rng(7)
    lm = torch.from_numpy(rng.normal(0.0, 0.3, (Z, net.R))).cuda()
    tz = torch.from_numpy(s["t_end"] * rng.uniform(0.1, 1.0, Z)).cuda()
    outs, grads = [], []
    for sp in ("generic", 2):
        tape = nb.Tape(nc, Z, 4000)
        out = nb.burn(nc, t["Y"], t["T9"], t["rho"], tz, s["rtol"], s["atol"], lm,
                      tape=tape, specialize=sp)
        torch.cuda.synchronize()
        assert int((out.status == 0).sum()) == Z
        gY = torch.zeros((1, Z, net.N), dtype=torch.float64, device="cuda")
        gY[0, :, 3] = 1.0
        gE = torch.ones((1, Z), dtype=torch.float64, device="cuda")
        g = nb.adjoint(nc, tape, gY, gE)
        torch.cuda.synchronize()
        outs.append(out)
        grads.append(g)
    _equal(outs[0], outs[1])
    for a, b in zip(grads[0], grads[1]):
        if a is not None:
            assert torch.equal(a, b)


def test_specialized_watchdog():
    # the watchdog lives in the shared claim loop: an exhausted budget ends
    # zones with TIMEOUT in the specialised kernel too
    nb, torch, net, z, s, t = _setup("chain13_heat", 4096)
    nc = nb.Network(net)
    out = nb.burn(nc, t["Y"], t["T9"], t["rho"], s["t_end"], s["rtol"], s["atol"],
                  specialize=1, time_budget_s=1e-9)
    torch.cuda.synchronize()
    st = out.status.cpu().numpy()
    assert (st == 6).sum() > 0
    done = st == 0
    ref = nb.burn(nc, t["Y"], t["T9"], t["rho"], s["t_end"], s["rtol"], s["atol"],
                  specialize="generic")
    torch.cuda.synchronize()
    assert torch.equal(out.Y[torch.from_numpy(done).cuda()],
                       ref.Y[torch.from_numpy(done).cuda()])


@pytest.mark.parametrize("name", ["chain13_heat", "chain13"])
def test_a_prepared_network_compiles_nothing_more(name):
    # after specialize() a default burn of any number of zones runs at once:
    # the ranges of its form are the number of zones an SM gets
    import time
    nb, torch, net, z, s, t = _setup(name, 20000)
    nc = nb.Network(net)
    nc.specialize()
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    a = lambda n: [t[k][:n].contiguous() for k in ("Y", "T9", "rho")]
    tol = (1e-9, s["rtol"], s["atol"])
    nb.zone_costs(nc, *a(20000), *tol)
    nb.burn(nc, *a(20000), *tol, specialize="generic")     # the device is warm
    torch.cuda.synchronize()
    for Z in (1, 12 * sm, 35 * sm, 58 * sm, 20000):
        start = time.perf_counter()
        nb.burn(nc, *a(Z), *tol)
        torch.cuda.synchronize()
        # a compilation takes seconds, these burns about a millisecond
        assert time.perf_counter() - start < 0.5
        assert nc.info()["last_specialized"] > 0


@pytest.mark.parametrize("name,warm", [("chain13_heat", 3000), ("chain13_heat", 20000),
                                       ("chain13", 1000)])
def test_a_captured_burn_takes_a_form_that_is_built(name, warm):
    # a burn of many zones, then the capture of one of few on the same
    # network: another form's range, with nothing to compile
    import time
    nb, torch, net, z, s, t = _setup(name, warm)
    nc = nb.Network(net)
    a = lambda n: [t[k][:n].contiguous() for k in ("Y", "T9", "rho")]
    tol = (1e-6, s["rtol"], s["atol"])
    full = nb.burn(nc, *a(warm), *tol)
    few = a(64)
    out = nb.burn(nc, *few, *tol, specialize="generic")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    start = time.perf_counter()
    with torch.cuda.graph(graph):
        nb.burn(nc, *few, *tol, out=out)
    assert time.perf_counter() - start < 1.0
    for x in out:
        x.zero_()
    graph.replay()
    torch.cuda.synchronize()
    for x, y in zip(out, full):
        assert torch.equal(x, y[:64])


@pytest.mark.parametrize("name,per_sm", [("chain13", 256), ("chain13", 160), ("chain13_heat", 200)])
def test_the_lane_kernels_block_fits_the_number_of_zones(name, per_sm):
    # the block chosen from the zones per SM against the others: within 12 %
    # of the best of them (all lanes at fixed temperature: 18 % slower)
    nb, torch, net, z, s, t = _setup(name, per_sm * 160)
    nc = nb.Network(net)
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    a = [t[k][:per_sm * sm].contiguous() for k in ("Y", "T9", "rho")]
    tol = (s["t_end"], s["rtol"], s["atol"])

    def ms(**kw):
        nb.burn(nc, *a, *tol, **kw)
        best = float("inf")
        for _ in range(3):
            x, y = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            x.record()
            nb.burn(nc, *a, *tol, **kw)
            y.record()
            y.synchronize()
            best = min(best, x.elapsed_time(y))
        return best

    shapes = [ms(specialize=3, threads_per_block=n) for n in (128, 160, 192, 256)]
    assert ms() < 1.12 * min(shapes)
