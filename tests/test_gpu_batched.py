"""Batched solver (many uneven problems in one cached CUDA-graph launch):
every problem's result equals the single-problem call bit for bit (same
kernels, same inputs), replays reuse the graph and see new data, AUTO
precisions are resolved per problem, and the results meet the solution
tolerance against the oracle."""
import ctypes as C
import threading

import numpy as np
import pytest
import torch

import oracle as O
import problems as P
from tests.gpu_util import assert_solution_parity, dev_colmajor, oracle_realizations, to_np

pytestmark = pytest.mark.gpu

lsq = pytest.importorskip("paper_2603_16644_gb300")


def make_batch(count, seed, auto=False):
    rng = np.random.default_rng(seed)
    probs, opts = [], []
    for i in range(count):
        n = int(rng.integers(16, 129))
        m = int(rng.integers(max(500, 4 * n), 5001))
        kap = float(10 ** rng.uniform(2, 8 if not auto else 10))
        rho = float(10 ** rng.uniform(-12, -2))
        pr = P.make_problem(m, n, kap, rho, seed * 1000 + i)
        kind = lsq.SPARSE_SIGN if i % 2 == 0 else lsq.GAUSSIAN
        s = (2 if i % 3 else 4) * n
        prec = lsq.AUTO if auto else [lsq.BF16, lsq.FP32, lsq.FP64, lsq.FP16][i % 4]
        opts.append(lsq.make_opts(kind=kind, s=s, zeta=min(8, s), seed=7 + i, sketch_prec=prec,
                                  qr_prec=lsq.FP64 if prec == lsq.FP64 else lsq.FP32, refine_steps=i % 2))
        probs.append(pr)
    return probs, opts


def test_batched_equals_single_calls_bitwise():
    probs, opts = make_batch(12, 1)
    As = [dev_colmajor(p.A) for p in probs]
    bs = [torch.from_numpy(p.b).cuda() for p in probs]
    xs = [torch.empty(p.shape[1], dtype=torch.float64, device="cuda") for p in probs]
    infos = [torch.zeros(1, dtype=torch.int32, device="cuda") for _ in probs]
    desc = lsq.batch_descriptors(As, bs, xs, infos, opts)
    ws = lsq.batched_workspace(desc)
    lsq.solve_batched(desc, ws)
    xb = [to_np(x).copy() for x in xs]
    for i, p in enumerate(probs):
        assert int(to_np(infos[i])[0]) == 0
        x1, info1 = lsq.pne(As[i], bs[i], opts=opts[i])
        np.testing.assert_array_equal(to_np(x1), xb[i])
    # replay (cached graph) gives the same bits; new data in the same buffers is used
    lsq.solve_batched(desc, ws)
    for i in range(len(probs)):
        np.testing.assert_array_equal(to_np(xs[i]), xb[i])
    bs[0].mul_(2.0)
    lsq.solve_batched(desc, ws)
    np.testing.assert_allclose(to_np(xs[0]), 2 * xb[0], rtol=1e-9)


@pytest.mark.parametrize("hpne", [False, True])
def test_batched_against_oracle(hpne):
    probs, opts = make_batch(6, 2)
    As = [dev_colmajor(p.A) for p in probs]
    bs = [torch.from_numpy(p.b).cuda() for p in probs]
    xs = [torch.empty(p.shape[1], dtype=torch.float64, device="cuda") for p in probs]
    infos = [torch.zeros(1, dtype=torch.int32, device="cuda") for _ in probs]
    desc = lsq.batch_descriptors(As, bs, xs, infos, opts)
    ws = lsq.batched_workspace(desc, hpne=hpne)
    lsq.solve_batched(desc, ws, hpne=hpne)
    for i, p in enumerate(probs):
        o = opts[i]
        ref = O.solve(p.A, p.b, hpne=hpne, kind=o.kind, s=o.s, zeta=o.zeta, seed=o.seed, sketch_prec=o.sketch_prec,
                      qr_prec=o.qr_prec, refine_steps=o.refine_steps)
        assert int(to_np(infos[i])[0]) == ref["info"] == 0
        more = oracle_realizations(p, hpne=hpne, kind=o.kind, s=o.s, zeta=o.zeta, seed=o.seed,
                                   sketch_prec=o.sketch_prec, qr_prec=o.qr_prec, refine_steps=o.refine_steps)
        assert_solution_parity(to_np(xs[i]), ref["x"], p.x_star, p.kappa, p.rho, f"problem {i}",
                               refined=o.refine_steps > 0, u_p=o.sketch_prec, realizations=more)


def test_batched_auto_precision_per_problem():
    probs, opts = make_batch(8, 3, auto=True)
    As = [dev_colmajor(p.A) for p in probs]
    bs = [torch.from_numpy(p.b).cuda() for p in probs]
    xs = [torch.empty(p.shape[1], dtype=torch.float64, device="cuda") for p in probs]
    infos = [torch.zeros(1, dtype=torch.int32, device="cuda") for _ in probs]
    desc = lsq.batch_descriptors(As, bs, xs, infos, opts)
    ws = lsq.batched_workspace(desc)
    lsq.solve_batched(desc, ws)
    for i in range(len(probs)):
        x1, _ = lsq.pne(As[i], bs[i], opts=opts[i])
        np.testing.assert_array_equal(to_np(x1), to_np(xs[i]))


def test_batched_bad_input():
    probs, opts = make_batch(2, 4)
    As = [dev_colmajor(p.A) for p in probs]
    bs = [torch.from_numpy(p.b).cuda() for p in probs]
    xs = [torch.empty(p.shape[1], dtype=torch.float64, device="cuda") for p in probs]
    infos = [torch.zeros(1, dtype=torch.int32, device="cuda") for _ in probs]
    opts[1].s = 1  # s < n
    desc = lsq.batch_descriptors(As, bs, xs, infos, opts)
    with pytest.raises(lsq.LsqError):
        lsq.batched_workspace(desc)
    with pytest.raises(lsq.LsqError):
        lsq.solve_batched(desc, torch.empty(1024, dtype=torch.uint8, device="cuda"))


def batch_buffers(probs, opts):
    As = [dev_colmajor(p.A) for p in probs]
    bs = [torch.from_numpy(p.b).cuda() for p in probs]
    xs = [torch.full((p.shape[1],), float("nan"), dtype=torch.float64, device="cuda") for p in probs]
    infos = [torch.full((1,), -9, dtype=torch.int32, device="cuda") for _ in probs]
    desc = lsq.batch_descriptors(As, bs, xs, infos, opts)
    return As, bs, xs, infos, desc, lsq.batched_workspace(desc)


def set_tc_sketch(on):
    f = lsq.lib().lsq_set_tensor_core_sketch
    f.restype = C.c_int32
    f.argtypes = [C.c_int32]
    return bool(f(int(on)))


@pytest.mark.parametrize("auto", [False, True])
@pytest.mark.parametrize("switch", [lsq.set_fp64_emulation, set_tc_sketch])
def test_batched_follows_the_switches(switch, auto):
    """The same descriptors after a switch was changed: the bits of single calls
    under the new setting, and of the old one once it is back."""
    probs, opts = make_batch(4, 21)
    for o in opts:
        o.kind, o.sketch_prec, o.qr_prec = lsq.GAUSSIAN, lsq.AUTO if auto else lsq.FP32, lsq.FP32
    As, bs, xs, infos, desc, ws = batch_buffers(probs, opts)
    for _ in range(3):  # enqueued, captured, replayed
        lsq.solve_batched(desc, ws)
    first = [to_np(x).copy() for x in xs]
    prev = switch(False)
    try:
        lsq.solve_batched(desc, ws)
        got = [to_np(x).copy() for x in xs]
        want = [to_np(lsq.pne(A, b, opts=o)[0]) for A, b, o in zip(As, bs, opts)]
    finally:
        switch(prev)
    for g, w in zip(got, want):
        np.testing.assert_array_equal(g, w)
    assert any(np.any(g != f) for g, f in zip(got, first))
    lsq.solve_batched(desc, ws)
    for x, f in zip(xs, first):
        np.testing.assert_array_equal(to_np(x), f)


def test_batched_follows_the_reduction_hook():
    """A hook set after a batch ran is called by the same batch's next run, and
    no more once it is removed."""
    probs, opts = make_batch(3, 22)
    As, bs, xs, infos, desc, ws = batch_buffers(probs, opts)
    for _ in range(3):  # enqueued, captured, replayed
        lsq.solve_batched(desc, ws)
    first = [to_np(x).copy() for x in xs]
    calls = []
    lsq.set_reduce_hook(lambda buf, count, kind, stream: calls.append(count) or 0)
    try:
        lsq.solve_batched(desc, ws)
        torch.cuda.synchronize()
    finally:
        lsq.set_reduce_hook(None)
    assert len(calls) >= 3 * len(probs)  # the sketch, the Gram and the right-hand side of each
    n = len(calls)
    lsq.solve_batched(desc, ws)
    assert len(calls) == n
    for x, f in zip(xs, first):
        np.testing.assert_array_equal(to_np(x), f)


def test_batched_launches_are_counted_once():
    """lsq_launch_count over a new batch is the sum over single calls (problems
    of one QR panel, where both run the same kernels), as over the call that captures
    it, also where it is enqueued and captured behind; a replay adds none."""
    probs, opts = [], []
    for i in range(3):
        probs.append(P.make_problem(900 + 100 * i, 30, 1e3, 1e-6, 77 + i))
        opts.append(lsq.make_opts(kind=lsq.SPARSE_SIGN, s=120, zeta=8, seed=i, sketch_prec=lsq.FP32))
    As, bs, xs, infos, desc, ws = batch_buffers(probs, opts)
    n0 = lsq.launch_count()
    for A, b, o in zip(As, bs, opts):
        lsq.pne(A, b, opts=o)
    n1 = lsq.launch_count()
    lsq.solve_batched(desc, ws)
    n2 = lsq.launch_count()
    assert n2 - n1 == n1 - n0 > 0
    lsq.solve_batched(desc, ws)
    assert lsq.launch_count() - n2 == n1 - n0
    n2 = lsq.launch_count()
    lsq.solve_batched(desc, ws)
    assert lsq.launch_count() == n2
    big = P.make_problem_torch(600000, 32, 1e3, 1e-6, 78)  # mean work above 1e9
    A, b = big[0], big[1]
    x, info = torch.zeros(32, dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    desc = lsq.batch_descriptors([A], [b], [x], [info], [lsq.make_opts(kind=lsq.SPARSE_SIGN, s=128, zeta=8, seed=1)])
    ws = lsq.batched_workspace(desc)
    count = []
    for _ in range(3):
        n0 = lsq.launch_count()
        lsq.solve_batched(desc, ws)
        count.append(lsq.launch_count() - n0)
    assert count[0] == count[1] > 0 == count[2]


@pytest.mark.parametrize("field,value", [("refine_steps", 2), ("qr_prec", lsq.BF16), ("row_offset", -1)])
def test_batched_refuses_before_any_problem_runs(field, value):
    """Options that a single call refuses, in a problem after heavier ones: the
    batch is refused with nothing launched, and runs without that problem."""
    probs, opts = make_batch(3, 23)
    probs.append(P.make_problem(600, 2, 10.0, 0.0, 5))
    opts.append(lsq.make_opts(kind=lsq.SPARSE_SIGN, s=20, zeta=4, seed=1, sketch_prec=lsq.FP32))
    As, bs, xs, infos, desc, ws = batch_buffers(probs, opts)
    setattr(desc[3].opts, field, value)
    n0 = lsq.launch_count()
    with pytest.raises(lsq.LsqError):
        lsq.solve_batched(desc, ws)
    assert lsq.launch_count() == n0
    for x, info in zip(xs, infos):
        assert np.isnan(to_np(x)).all() and int(to_np(info)[0]) == -9
    three = lsq.batch_descriptors(As[:3], bs[:3], xs[:3], infos[:3], opts[:3])
    lsq.solve_batched(three, ws)
    for A, b, x, o in zip(As, bs, xs[:3], opts):
        np.testing.assert_array_equal(to_np(x), to_np(lsq.pne(A, b, opts=o)[0]))


def test_batched_sketch_refuses_the_transform_order_before_any_runs():
    """An SRFT of more rows than the transform takes (2^22 in FP32)."""
    big = torch.randn((1, 2**22 + 1), dtype=torch.float64, device="cuda").t()
    small = dev_colmajor(np.random.default_rng(1).standard_normal((4000, 200)))
    ob = lsq.make_opts(kind=lsq.SRFT, s=8, zeta=0, seed=1, sketch_prec=lsq.FP32)
    os_ = lsq.make_opts(kind=lsq.GAUSSIAN, s=4000, zeta=0, seed=1, sketch_prec=lsq.FP32)
    n0 = lsq.launch_count()
    with pytest.raises(lsq.LsqError):
        lsq.sketch_batched([small, big], [os_, ob])
    assert lsq.launch_count() == n0


def test_new_batches_in_a_row_without_synchronisation():
    """Batches never seen before, one after another on one stream and on two,
    each enqueued while the ones before still run; then each three times in a row
    (enqueued, captured, replayed), again without waiting, and in turn once more:
    the bits of single calls."""
    sets = []
    for k in range(4):
        probs, opts = make_batch(5, 30 + k)
        sets.append((opts, batch_buffers(probs, opts)))
    want = [[to_np(lsq.pne(A, b, opts=o)[0]).copy() for A, b, o in zip(bufs[0], bufs[1], opts)] for opts, bufs in sets]
    other = torch.cuda.Stream()
    for streams, calls in [([None] * 4, 1), ([None, other] * 2, 1), ([None] * 4, 3), ([None, other] * 2, 3), ([None] * 4, 1)]:
        for _, bufs in sets:
            for x in bufs[2]:
                x.fill_(float("nan"))
        torch.cuda.synchronize()
        for st, (_, bufs) in zip(streams, sets):
            with torch.cuda.stream(st):
                for _ in range(calls):
                    lsq.solve_batched(bufs[4], bufs[5])
        torch.cuda.synchronize()
        for (_, bufs), ws in zip(sets, want):
            for x, w, info in zip(bufs[2], ws, bufs[3]):
                assert int(to_np(info)[0]) == 0
                np.testing.assert_array_equal(to_np(x), w)


def test_new_batches_from_two_threads():
    """Two threads, each with a stream and two batches of its own, one of them
    three times in a row, so that calls meet the other thread's graph in the cache."""
    work = []
    for t in range(2):
        mine = []
        for k in range(2):
            probs, opts = make_batch(3, 40 + 2 * t + k)
            bufs = batch_buffers(probs, opts)
            mine.append((bufs, [to_np(lsq.pne(A, b, opts=o)[0]).copy() for A, b, o in zip(bufs[0], bufs[1], opts)]))
        work.append(mine)
    torch.cuda.synchronize()
    bad = []

    def run(mine):
        try:
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                for _ in range(3):
                    for bufs, want in [mine[0]] * 3 + [mine[1]]:
                        for x in bufs[2]:
                            x.fill_(float("nan"))
                        lsq.solve_batched(bufs[4], bufs[5])
                        st.synchronize()
                        for x, w in zip(bufs[2], want):
                            if not np.array_equal(x.cpu().numpy(), w):
                                bad.append("bits")
        except Exception as e:
            bad.append(repr(e))

    threads = [threading.Thread(target=run, args=(m,)) for m in work]
    for th in threads:
        th.start()
    for th in threads:
        th.join(120)
        assert not th.is_alive()
    assert not bad, bad


def test_autotuner_picks_a_candidate(tmp_path):
    from paper_2603_16644_gb300.autotune import CANDIDATES, Autotuner

    tuner = Autotuner(path=str(tmp_path / "tune.json"))
    kind, s = tuner.choose(3000, 100, prec=lsq.FP32)
    assert (kind, s // 100) in CANDIDATES
    again = Autotuner(path=str(tmp_path / "tune.json"))
    assert again.choose(3000, 100, prec=lsq.FP32) == (kind, s)


def test_batched_sketch_and_qr_equal_single_calls():
    # lsq_sketch_batched / lsq_precond_qr_batched: one captured fan-out, the
    # results of separate calls bit for bit
    rng = np.random.default_rng(9)
    As, opts = [], []
    for i in range(10):
        n = int(rng.integers(8, 200))
        m = int(rng.integers(4 * n, 6000))
        A = dev_colmajor(np.asfortranarray(rng.standard_normal((m, n)) * np.exp2(rng.integers(-8, 8, n))[None, :]))
        kind = lsq.SPARSE_SIGN if i % 2 else lsq.GAUSSIAN
        prec = [lsq.FP8_E4M3, lsq.BF16, lsq.FP16, lsq.FP32, lsq.FP64][i % 5]
        As.append(A)
        opts.append(lsq.make_opts(kind=kind, s=(2 + i % 3) * n, zeta=min(8, 2 * n), seed=100 + i, sketch_prec=prec))
    outs = lsq.sketch_batched(As, opts)
    for A, o, (Asb, ceb, infob) in zip(As, opts, outs):
        As1, ce1, info1 = lsq.sketch(A, o)
        assert int(to_np(infob)[0]) == int(to_np(info1)[0]) == 0
        np.testing.assert_array_equal(to_np(Asb), to_np(As1))
        np.testing.assert_array_equal(to_np(ceb), to_np(ce1))
    qr = lsq.precond_qr_batched([(Asb, ceb) for Asb, ceb, _ in outs])
    for (Asb, ceb, _), (Rb, infob), o in zip(outs, qr, opts):
        qp = lsq.FP64 if o.sketch_prec == lsq.FP64 else lsq.FP32
        R1, info1 = lsq.precond_qr(Asb, ceb, qp)
        assert int(to_np(infob)[0]) == int(to_np(info1)[0]) == 0
        np.testing.assert_array_equal(np.triu(to_np(Rb)), np.triu(to_np(R1)))


def test_batched_auto_sketch_per_problem():
    probs, opts = make_batch(8, 5, auto=True)
    for o in opts:
        o.sketch_prec = lsq.AUTO_SKETCH
    As = [dev_colmajor(p.A) for p in probs]
    bs = [torch.from_numpy(p.b).cuda() for p in probs]
    xs = [torch.empty(p.shape[1], dtype=torch.float64, device="cuda") for p in probs]
    infos = [torch.zeros(1, dtype=torch.int32, device="cuda") for _ in probs]
    desc = lsq.batch_descriptors(As, bs, xs, infos, opts)
    ws = lsq.batched_workspace(desc)
    lsq.solve_batched(desc, ws)
    for i in range(len(probs)):
        x1, _ = lsq.pne(As[i], bs[i], opts=opts[i])
        np.testing.assert_array_equal(to_np(x1), to_np(xs[i]))


def test_batched_full_size_uneven_batch():
    # the batched workload at full size: 512 problems, m uniform in [2000, 40000],
    # n uniform in [32, 512], kappa log-uniform in [1e2, 1e10], relative
    # residual log-uniform in [1e-12, 1e-2]; sketch kind and s in {2n, 4n} from
    # the autotuner, precision per problem from the estimate on a sketch
    from types import SimpleNamespace

    from paper_2603_16644_gb300.autotune import Autotuner

    rng = np.random.default_rng(2603)
    tuner = Autotuner()
    As, bs, xs, infos, opts, meta = [], [], [], [], [], []
    for i in range(512):
        n = int(rng.integers(32, 513))
        m = int(rng.integers(max(2000, 4 * n), 40001))
        kap = float(10 ** rng.uniform(2, 10))
        rho = float(10 ** rng.uniform(-12, -2))
        seed = P.seed_for(3, i)
        A, b, x_star, _, _ = P.make_problem_torch(m, n, kap, rho, seed)
        kind, s = tuner.choose(m, n, prec=lsq.FP32)
        As.append(A)
        bs.append(b)
        xs.append(torch.empty(n, dtype=torch.float64, device="cuda"))
        infos.append(torch.zeros(1, dtype=torch.int32, device="cuda"))
        opts.append(lsq.make_opts(kind=kind, s=s, zeta=min(8, s), seed=seed, sketch_prec=lsq.AUTO_SKETCH,
                                  qr_prec=lsq.FP32, refine_steps=0))
        meta.append((kap, rho, x_star))
    desc = lsq.batch_descriptors(As, bs, xs, infos, opts)
    ws = lsq.batched_workspace(desc)
    lsq.solve_batched(desc, ws)  # estimate pass, capture, first launch
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    lsq.solve_batched(desc, ws)  # estimate pass and one cached graph launch
    e1.record()
    torch.cuda.synchronize()
    print(f"512 uneven problems: {512 / (e0.elapsed_time(e1) / 1000):.1f} solves/s")
    assert all(int(to_np(f)[0]) == 0 for f in infos)
    # bit-identical to single calls on a sample
    for i in range(0, 512, 37):
        x1, _ = lsq.pne(As[i], bs[i], opts=opts[i])
        np.testing.assert_array_equal(to_np(x1), to_np(xs[i]))
    # against the oracle on a subset, at the precision the estimate chose
    for i in range(3, 512, 16):
        kap, rho, x_star = meta[i]
        _, ch = lsq.condest_sketch(As[i], seed=opts[i].seed)
        prec = int(to_np(ch)[0])
        A_np, b_np = to_np(As[i]), to_np(bs[i])
        kw = dict(kind=opts[i].kind, s=opts[i].s, zeta=opts[i].zeta, seed=opts[i].seed, sketch_prec=prec,
                  qr_prec=O.FP64 if prec == O.FP64 else O.FP32, refine_steps=0)
        ref = O.solve(A_np, b_np, **kw)
        assert ref["info"] == 0
        more = oracle_realizations(SimpleNamespace(A=A_np, b=b_np), **kw)
        assert_solution_parity(to_np(xs[i]), ref["x"], to_np(x_star), kap, rho, f"problem {i}", refined=False,
                               u_p=prec, realizations=more)
