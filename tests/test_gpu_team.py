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


@pytest.mark.parametrize("name", ["chain13", "chain13_heat", "chain13_heat_ap",
                                  "chain13_heat_scr", "chain13_heat_tab", "chain13_literal"])
def test_generated_teams_give_the_lane_kernels_bits(name):
    # the generated kernel's team forms (32, 16, 8, 4 lanes a zone, by zones per
    # SM) against one zone per lane, on both sides of every line of the rule
    nb, torch, net, t, tol, sm = _setup(name, 11600, 1e-6)
    kw = lambda n: dict(zeta=t["zeta"][:n].contiguous()) if "zeta" in t else {}
    ref = nb.burn(net, *_first(t, 11600), *tol, specialize="generic", **kw(11600))
    assert net.info()["last_specialized"] == 0
    for Z in (1, 33, 5 * sm, 5 * sm + 1, 12 * sm, 12 * sm + 1, 35 * sm + 1, 40 * sm + 1, 60 * sm,
              60 * sm + 1, 72 * sm + 1):
        out = nb.burn(net, *_first(t, Z), *tol, **kw(Z))
        assert net.info()["last_specialized"] > 0
        _same(torch, out, ref, Z)


def test_generated_teams_with_options_tape_and_watchdog():
    nb, torch, net, t, tol, sm = _setup("chain13_heat", 2 * 160, 1e-6)
    Z = 320
    rng = np.random.default_rng(9)
    lm = torch.from_numpy(rng.normal(0.0, 0.3, (Z, net.R))).cuda()
    tz = torch.from_numpy(1e-6 * rng.uniform(0.0, 1.0, Z)).cuda()
    tz[3] = 0.0
    outs, grads = [], []
    for sp in ("generic", 0):
        tape = nb.Tape(net, Z, 900)
        outs.append(nb.burn(net, *_first(t, Z), tz, tol[1], tol[2], lm, tape=tape, specialize=sp))
        gY = torch.ones((1, Z, net.N), dtype=torch.float64, device="cuda")
        grads.append(nb.adjoint(net, tape, gY))
    _same(torch, outs[0], outs[1], Z)
    for a, b in zip(*grads):
        assert torch.equal(a, b)
    out = nb.burn(net, *_first(t, Z), *tol, max_attempts=20)
    ref = nb.burn(net, *_first(t, Z), *tol, max_attempts=20, specialize="generic")
    _same(torch, out, ref, Z)
    assert int((out.status == 1).sum()) > 0
    out = nb.burn(net, *_first(t, Z), 1e-3, tol[1], tol[2], time_budget_s=1e-9)
    assert int((out.status == 6).sum()) == Z


def test_last_zones_move_between_warps_with_the_same_bits():
    # a block's last zones are packed into fewer warps, with and without more
    # zones than lanes
    nb, torch, net, t, tol, sm = _setup("chain13_heat", 70000, 1e-7)
    ref = nb.burn(net, *_first(t, 70000), *tol, kernel="plain")
    for tpb, bps, n in ((256, 1, 70000), (64, 2, 30011), (160, 1, 5003)):
        out = nb.burn(net, *_first(t, n), *tol, specialize=3, threads_per_block=tpb,
                      blocks_per_sm=bps, schedule="fifo")
        _same(torch, out, ref, n)
    fixed = nb.Network(gen.network("chain13"))
    z = gen.zones("chain13", 3000)
    a = [torch.from_numpy(z[k]).cuda() for k in ("Y", "T9", "rho")]
    ref = nb.burn(fixed, *a, 1e-6, 1e-8, 1e-12, kernel="plain")
    for v in (1, 2, 3):
        out = nb.burn(fixed, *a, 1e-6, 1e-8, 1e-12, specialize=v, threads_per_block=256)
        _same(torch, out, ref, 3000)


@pytest.mark.parametrize("name,K,t_end,big", [("chain13_heat", 2, 1e-6, 4000),
                                              ("chain13", 1, 1e-6, 25000),
                                              ("chain13_heat_tab", 9, 1e-6, 400),
                                              ("net48_adjoint", 2, 1e-5, 70)])
def test_lane_tapes_by_teams_give_the_lane_adjoints_bits(name, K, t_end, big):
    # a launch shape asked for runs the lane kernel; without one the teams'
    # lanes follow the zones per SM
    nb, torch, net, t, tol, sm = _setup(name, big, t_end)
    rng = np.random.default_rng(5)
    for Z in sorted({Z for Z in (1, 33, 12 * sm, 12 * sm + 1, 24 * sm + 1, big) if Z <= big}):
        lm = torch.from_numpy(rng.normal(0.0, 0.1, net.R)).cuda()
        tape = nb.Tape(net, Z, 1000)
        out = nb.burn(net, *_first(t, Z), *tol, lm, tape=tape)
        assert int((out.status == 0).sum()) == Z
        gY = torch.from_numpy(rng.normal(size=(K, Z, net.N))).cuda()
        gE = torch.from_numpy(rng.normal(size=(K, Z))).cuda()
        gT = torch.from_numpy(rng.normal(size=(K, Z))).cuda()
        ref = nb.adjoint(net, tape, gY, gE, gT, kernel="persistent", threads_per_block=32)
        for a, b in zip(nb.adjoint(net, tape, gY, gE, gT), ref):
            assert torch.equal(a, b)


def test_several_networks_by_teams_give_single_burns_bits():
    # the lanes per zone follow all sets' zones; with a large network a warp
    nb, torch, _, t, tol, sm = _setup("chain13_heat", 6000, 1e-7)
    nets = [nb.Network(gen.network(n)) for n in ("chain13_heat", "chain13", "chain13_heat_ap")]
    lanes = dict(threads_per_block=64, specialize="generic")

    def check(sets):
        for d, out in zip(sets, nb.burn_multi(sets, *tol)):
            ref = nb.burn(d["net"], d["Y0"], d["T9"], d["rho"], *tol, **lanes)
            _same(torch, out, ref, d["Y0"].shape[0])

    def chain(net, n):
        return dict(zip(("Y0", "T9", "rho"), _first(t, n)), net=net)

    for Z in (1, 5 * sm // 3 + 1, 12 * sm // 3 + 1):
        check([chain(n, Z) for n in nets])
    check([chain(n, 5600) for n in nets])     # beyond 100 zones an SM: the lane kernel
    big, z, _ = gen.problem("net48", 40)
    a = {k: torch.from_numpy(z[q]).cuda() for k, q in (("Y0", "Y"), ("T9", "T9"), ("rho", "rho"))}
    check([chain(nets[0], 100), dict(a, net=nb.Network(big))])


@pytest.mark.parametrize("name,Z,t_end", [("net48", 1, 1e-5), ("net48", 1000, 1e-6),
                                          ("net128_heat", 33, 1e-8)])
def test_large_networks_by_lane_order_teams_give_the_lane_kernels_bits(name, Z, t_end):
    nb, torch, net, t, tol, sm = _setup(name, Z, t_end)
    ref = nb.burn(net, *_first(t, Z), *tol, threads_per_block=32)
    for kw in (dict(), dict(specialize="generic"), dict(schedule="fifo")):
        _same(torch, nb.burn(net, *_first(t, Z), *tol, **kw), ref, Z)


@pytest.mark.parametrize("kw", [dict(max_attempts=1), dict(max_attempts=7),
                                dict(max_attempts=300)])
def test_zones_of_a_block_that_end_at_once(kw):
    # all zones of a warp reach the attempt limit in the same turn, while
    # other warps' zones end earlier or have ended
    nb, torch, net, t, tol, sm = _setup("chain13_heat", 20000)
    ref = nb.burn(net, *_first(t, 20000), *tol, kernel="plain", **kw)
    assert int((ref.status == 1).sum()) > 0
    for tpb, n in ((256, 20000), (160, 20000), (64, 700)):
        out = nb.burn(net, *_first(t, n), *tol, specialize=3, threads_per_block=tpb, **kw)
        _same(torch, out, ref, n)


@pytest.mark.parametrize("K", [1, 2])
def test_large_networks_lane_tapes_beyond_a_zone_an_sm(K):
    # a team of two warps is a block of its own, however many zones an SM gets
    nb, torch, net, t, tol, sm = _setup("net48_adjoint", 3 * 160 + 1, 1e-6)
    rng = np.random.default_rng(8)
    for Z in (sm, sm + 1, 3 * sm):
        tape = nb.Tape(net, Z, 400)
        nb.burn(net, *_first(t, Z), *tol, tape=tape)
        gY = torch.from_numpy(rng.normal(size=(K, Z, net.N))).cuda()
        gE = torch.from_numpy(rng.normal(size=(K, Z))).cuda()
        ref = nb.adjoint(net, tape, gY, gE, kernel="persistent", threads_per_block=32)
        for a, b in zip(nb.adjoint(net, tape, gY, gE), ref):
            assert torch.equal(a, b)


@pytest.mark.parametrize("call", ["burn", "coop", "adjoint", "multi"])
def test_networks_of_different_sizes_from_two_threads(call):
    # each thread its own network and stream; the kernels are the same, their
    # shared memory differs from network to network
    import threading
    nb, torch, *_ = _setup("chain13", 1)
    ref, got, errors = {}, {}, []

    def work(name, Z, rounds, into):
        _, _, net, t, tol, _ = _setup(name, Z, 1e-12)
        a = _first(t, Z)
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            stream.wait_stream(torch.cuda.default_stream())
            for _ in range(rounds):
                if call == "multi":
                    out = nb.burn_multi([dict(net=net, Y0=a[0], T9=a[1], rho=a[2])], *tol)[0]
                elif call == "adjoint":
                    tape = nb.Tape(net, Z, 50)
                    nb.burn(net, *a, *tol, tape=tape)
                    out = nb.adjoint(net, tape, torch.ones((1, Z, net.N), dtype=torch.float64,
                                                           device="cuda"))
                else:
                    out = nb.burn(net, *a, *tol,
                                  kernel="coop" if call == "coop" else "persistent")
        stream.synchronize()
        into[name] = out

    def guarded(*args):
        try:
            work(*args)
        except Exception as e:      # a refused launch
            errors.append(e)

    pairs = (("net48", 8), ("net128_heat", 8))
    for name, Z in pairs:
        work(name, Z, 1, ref)
    threads = [threading.Thread(target=guarded, args=(name, Z, 400, got)) for name, Z in pairs]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors
    for name, _ in pairs:
        for a, b in zip(got[name], ref[name]):
            assert torch.equal(a, b)


def test_a_blob_and_a_zone_that_just_fit_shared_memory():
    # 202,560 bytes of compiled network and 29,808 of one zone's arrays of the
    # 232,448 a block may have; a team's arrays are 144 bytes more
    import dataclasses
    import paper_2312_02836_gb300 as nb
    import torch
    from gen import workloads as wl
    N = 68
    rng = np.random.Generator(np.random.PCG64(31))
    reac, prod = wl._random_topology(rng, N, (81, 136, 27))
    keep = np.arange(reac.shape[0]) != 8
    spec = dataclasses.replace(gen.network("net48"), N=N, R=int(keep.sum()),
                               reactants=reac[keep], products=prod[keep],
                               A=np.arange(1, N + 1, dtype=np.float64),
                               coeffs=wl._draw_coeffs(rng, reac.shape[0])[keep])
    net = nb.Network(spec)
    Z = 40
    Y = np.zeros((Z, N))
    Y[:, :4] = gen.zones("net48", Z)["Y"][:, :4]
    a = [torch.from_numpy(x).cuda() for x in (Y, gen.zones("net48", Z)["T9"],
                                              gen.zones("net48", Z)["rho"])]
    tol = (1e-6, 1e-8, 1e-12)
    ref = nb.burn(net, *a, *tol, kernel="coop")
    for tpb in (0, 32):
        out = nb.burn(net, *a, *tol, kernel="coop", blob_in_shared=1, threads_per_block=tpb)
        _same(torch, out, ref, Z)
    for wpz in (2, 4):
        nb.burn(net, *a, *tol, kernel="coop", blob_in_shared=1, warps_per_zone=wpz)
    with pytest.raises(nb.NetburnError):       # two zones never fitted
        nb.burn(net, *a, *tol, kernel="coop", blob_in_shared=1, threads_per_block=64)


def test_a_large_networks_blob_asked_for_in_shared_memory():
    # 48 species fit (the lane kernel), 128 don't
    nb, torch, net, t, tol, sm = _setup("net48", 8, 1e-7)
    ref = nb.burn(net, *_first(t, 8), *tol)
    _same(torch, nb.burn(net, *_first(t, 8), *tol, blob_in_shared=1), ref, 8)
    _, _, net, t, tol, _ = _setup("net128_heat", 8, 1e-9)
    nb.burn(net, *_first(t, 8), *tol)
    with pytest.raises(nb.NetburnError):
        nb.burn(net, *_first(t, 8), *tol, blob_in_shared=1)


@pytest.mark.parametrize("N,mix,heat", [(22, (19, 32, 6), True), (28, (30, 50, 10), True),
                                        (28, (30, 50, 10), False)])
def test_generated_teams_of_middle_networks(N, mix, heat):
    # networks between the chain and 48 species: fewer teams fit a block, and
    # few of them an SM
    import paper_2312_02836_gb300 as nb
    import torch
    from tests.test_codegen import _random_network
    net = nb.Network(_random_network(N, mix, heat))
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    Z = 61 * sm
    rng = np.random.default_rng(N)
    Y = np.zeros((Z, N))
    Y[:, :4] = rng.dirichlet([0.3] * 4, Z) / np.arange(1, 5)
    log_u = lambda lo, hi: np.exp(rng.uniform(np.log(lo), np.log(hi), Z))
    t = {k: torch.from_numpy(v).cuda()
         for k, v in (("Y", Y), ("T9", log_u(0.5, 4.0)), ("rho", log_u(1e5, 1e7)))}
    tol = (1e-4, 1e-8, 1e-12)
    ref = nb.burn(net, *_first(t, Z), *tol, specialize="generic", threads_per_block=64)
    assert int((ref.status == 0).sum()) == Z
    for n in (1, 5 * sm, 12 * sm, 35 * sm, 60 * sm, Z):
        out = nb.burn(net, *_first(t, n), *tol)
        assert net.info()["last_specialized"] > 0
        _same(torch, out, ref, n)


def _best_ms(torch, call, n=3):
    call()
    ms = []
    for _ in range(n):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        call()
        b.record()
        b.synchronize()
        ms.append(a.elapsed_time(b))
    return min(ms)


@pytest.mark.parametrize("name,per_sm", [("chain13", 32), ("chain13", 33), ("chain13", 40),
                                         ("chain13_heat", 60), ("chain13_heat_ap", 68)])
def test_teams_are_no_slower_than_the_lanes_they_replace(name, per_sm):
    # 15 % for the noise; teams past their line were 28 % slower
    nb, torch, net, t, tol, sm = _setup(name, per_sm * 160)
    a = _first(t, per_sm * sm)
    lane = _best_ms(torch, lambda: nb.burn(net, *a, *tol, specialize=3,
                                           threads_per_block=(per_sm + 31) // 32 * 32))
    assert _best_ms(torch, lambda: nb.burn(net, *a, *tol)) < 1.15 * lane


@pytest.mark.parametrize("name,Z", [("chain13_heat", 6), ("net48", 12)])
def test_cooperative_shapes_hold_the_zones_they_ask_for(name, Z):
    # small networks keep a warp a zone; an explicit shape counts a warp a zone
    # whatever the team: all zones of an SM at once take little longer than one
    # (in turns they took three times as long)
    nb, torch, net, t, tol, sm = _setup(name, Z * 160, 1e-4 if name == "net48" else None)
    a = _first(t, Z * sm)
    hard = int(nb.burn(net, *a, *tol, kernel="coop").counters[:, :3].sum(1).argmax())
    one = [x[hard:hard + 1].contiguous() for x in a]
    kw = dict(kernel="coop", threads_per_block=128, blocks_per_sm=3)
    alone = _best_ms(torch, lambda: nb.burn(net, *one, *tol, **kw))
    assert _best_ms(torch, lambda: nb.burn(net, *a, *tol, **kw)) < 2.0 * alone


def test_cooperative_shape_of_one_block_an_sm():
    # 128 threads, one block: four zones an SM at a time, not one team
    nb, torch, net, t, tol, sm = _setup("net48", 4 * 160, 1e-4)
    a = _first(t, 4 * sm)
    shape = lambda bps: _best_ms(torch, lambda: nb.burn(
        net, *a, *tol, kernel="coop", threads_per_block=128, blocks_per_sm=bps))
    assert shape(1) < 1.4 * shape(3)


@pytest.mark.parametrize("K,stride,per_sm", [(1, 64, 100), (1, 256, 20), (1, 256, 60),
                                             (9, 256, 100), (1, 1000, 100), (1, 0, 150)])
def test_lane_adjoint_by_teams_is_no_slower_whatever_the_tape(K, stride, per_sm):
    # a longer checkpoint stride and more cotangents leave room for fewer teams
    # (15 % for the noise; without the rule up to five times the lanes' time)
    nb, torch, net, t, tol, sm = _setup("chain13_heat", per_sm * 160, 1e-5)
    Z = per_sm * sm
    tape = nb.Tape(net, Z, 1000, stride)
    nb.burn(net, *_first(t, Z), *tol, tape=tape)
    rng = np.random.default_rng(4)
    gY = torch.from_numpy(rng.normal(size=(K, Z, net.N))).cuda()
    lane = dict(kernel="persistent", threads_per_block=max(32, per_sm // 32 * 32),
                blocks_per_sm=2)
    for a, b in zip(nb.adjoint(net, tape, gY), nb.adjoint(net, tape, gY, **lane)):
        assert torch.equal(a, b)
    ref = _best_ms(torch, lambda: nb.adjoint(net, tape, gY, **lane), 2)
    assert _best_ms(torch, lambda: nb.adjoint(net, tape, gY), 2) < 1.15 * ref


def test_cooperative_adjoint_of_small_networks_holds_an_sms_zones():
    # a warp a zone: eight zones an SM take little longer than one (four warps
    # a zone, two of them at a time: three times)
    nb, torch, net, t, tol, sm = _setup("chain13_heat", 8 * 160, 1e-4)

    def ms(Z):
        tape = nb.Tape(net, Z, 1400)
        nb.burn(net, *_first(t, Z), *tol, kernel="coop", tape=tape)
        gY = torch.ones((1, Z, net.N), dtype=torch.float64, device="cuda")
        return _best_ms(torch, lambda: nb.adjoint(net, tape, gY), 2)

    assert ms(8 * sm) < 2.0 * ms(sm)


def test_cooperative_adjoint_bits_of_a_middle_network():
    import paper_2312_02836_gb300 as nb
    import torch
    from tests.test_codegen import _random_network
    net = nb.Network(_random_network(28, (30, 50, 10), True))
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    Z, K = 8 * sm + 1, 3
    rng = np.random.default_rng(2)
    Y = np.zeros((Z, 28))
    Y[:, :4] = rng.dirichlet([0.3] * 4, Z) / np.arange(1, 5)
    log_u = lambda lo, hi: np.exp(rng.uniform(np.log(lo), np.log(hi), Z))
    t = {k: torch.from_numpy(v).cuda()
         for k, v in (("Y", Y), ("T9", log_u(0.5, 4.0)), ("rho", log_u(1e5, 1e7)))}
    gY = torch.from_numpy(rng.normal(size=(K, Z, 28))).cuda()

    def grads(n, **kw):
        tape = nb.Tape(net, n, 600)
        nb.burn(net, *_first(t, n), 1e-5, 1e-8, 1e-12, kernel="coop", tape=tape)
        return nb.adjoint(net, tape, gY[:, :n].contiguous(), kernel="coop", **kw)

    full = grads(Z)
    for n, kw in ((8 * sm, {}), (5, {}), (Z, dict(threads_per_block=128, blocks_per_sm=1)),
                  (Z, dict(ws_in_shared=0))):
        for a, b in zip(grads(n, **kw), full):
            assert torch.equal(a, b[:, :n])


def test_an_explicit_cooperative_block_leaves_the_blob_out():
    # 36 species: 96,304 bytes of compiled network, which the library keeps in
    # shared memory by itself, and eight zones of 17,392 don't fit a block
    # together; the zones alone do
    import paper_2312_02836_gb300 as nb
    import torch
    from tests.test_codegen import _random_network
    net = nb.Network(_random_network(36, (50, 83, 16), True))
    Z = 100
    rng = np.random.default_rng(6)
    Y = np.zeros((Z, 36))
    Y[:, :4] = rng.dirichlet([0.3] * 4, Z) / np.arange(1, 5)
    a = [torch.from_numpy(x).cuda() for x in (Y, rng.uniform(0.5, 3.0, Z),
                                              np.exp(rng.uniform(np.log(1e5), np.log(1e7), Z)))]
    tol = (1e-5, 1e-8, 1e-12)
    ref = nb.burn(net, *a, *tol, kernel="coop")
    for kw in (dict(threads_per_block=256), dict(threads_per_block=256, blocks_per_sm=1),
               dict(threads_per_block=32, blob_in_shared=1)):
        _same(torch, nb.burn(net, *a, *tol, kernel="coop", **kw), ref, Z)
    with pytest.raises(nb.NetburnError):
        nb.burn(net, *a, *tol, kernel="coop", threads_per_block=256, blob_in_shared=1)
