"""GPU parity of the whole-step persistent launch (rwkvq_step_plan / rwkvq_step_run) against the
oracle, product by product."""
import numpy as np
import pytest
import torch

from paper_2505_03803_b200 import binding as B
from paper_2505_03803_b200 import inputs
from tests import helpers as H

pytestmark = pytest.mark.gpu


def _build_ops(d, h, layers, Bn, bits, seed, all_method=None):
    """Logical codes drawn at random (valid by construction), packed by the library."""
    ops = []
    k = 0
    for l in range(layers):
        for (name, oc, ic, has_mu, stage) in inputs.layer_shapes(d, h):
            k += 1
            use_sq = (k % 3 != 0) if all_method is None else (all_method == B.RWKVQ_SQ)
            W = H.pack_sq(H.random_sq_codes(seed + k, oc, ic)) if use_sq else H.pack_vq(H.random_vq_codes(seed + k, oc, ic, bits), bits)
            mu = H.pack_mu(H.random_mu_codes(seed + 100 + k, ic, bits), bits) if has_mu else None
            x, xp = inputs.gen_activation_pair(seed + 200 + k, Bn, ic, n_outliers=4)
            x16, xp16 = x.astype(np.float16), xp.astype(np.float16)
            e = dict(W=W, mu=mu, x16=x16, xp16=xp16, stage=4 * l + stage,
                     xd=torch.from_numpy(x16).cuda(), xpd=torch.from_numpy(xp16).cuda() if has_mu else None,
                     y=torch.full((Bn, oc), float("nan"), dtype=torch.float32, device="cuda"))
            ops.append(e)
    ops.sort(key=lambda e: e["stage"])
    return ops


def _plan(ops, Bn):
    arr = B.make_ops([dict(desc=e["W"].desc, W=e["W"].dev, mu_desc=None if e["mu"] is None else e["mu"].desc,
                           mu=None if e["mu"] is None else e["mu"].dev, x=e["xd"], xprev=e["xpd"], y=e["y"],
                           stage=e["stage"]) for e in ops])
    n = B.rwkvq_step_plan_bytes(arr, Bn)
    assert n > 0
    plan = torch.zeros(n, dtype=torch.uint8, device="cuda")
    B.rwkvq_step_plan(arr, Bn, plan)
    return plan


def _forms(ops, Bn):
    return B.rwkvq_step_plan_forms(ops, Bn, torch.cuda.get_device_properties(0).multi_processor_count)


def _check(ops, Bn):
    worst = 0.0
    for e in ops:
        y = e["y"].double().cpu().numpy()
        ref, tol = H.reference(e["W"], e["mu"], e["x16"], e["xp16"])
        err = np.abs(y - ref)
        assert np.isfinite(y).all()
        ratio = float((err / tol).max())
        worst = max(worst, ratio)
        assert (err <= tol).all(), f"stage {e['stage']}: max err/tol = {ratio}"
    return worst


@pytest.mark.parametrize("Bn,bits", [(1, 6), (8, 6), (16, 8), (3, 8), (2, 6), (4, 6), (7, 8), (9, 6), (12, 8)])
def test_step_matches_oracle_small_stack(Bn, bits):
    ops = _build_ops(512, 1280, 2, Bn, bits, seed=10 * Bn + bits)   # h = 5 column tiles: odd tile count
    plan = _plan(ops, Bn)
    for rep in range(3):          # outputs are cleared and recomputed on every run
        B.rwkvq_step_run(plan)
        torch.cuda.synchronize()
        assert B.rwkvq_device_status() == 0
        _check(ops, Bn)


@pytest.mark.parametrize("method", [B.RWKVQ_SQ, B.RWKVQ_VQ])
def test_step_matches_oracle_1p6b_layer(method):
    ops = _build_ops(2048, 7168, 1, 1, 6, seed=77, all_method=method)
    plan = _plan(ops, 1)
    B.rwkvq_step_run(plan)
    torch.cuda.synchronize()
    assert B.rwkvq_device_status() == 0
    _check(ops, 1)


@pytest.mark.parametrize("Bn", [1, 5, 16])
def test_step_ragged_sq_shapes(Bn):
    # d = 384, h = 896: row counts that end in a half unit (one 128-row chunk) and input lengths
    # whose last 256-column tile is half empty
    ops = _build_ops(384, 896, 2, Bn, 6, seed=300 + Bn, all_method=B.RWKVQ_SQ)
    plan = _plan(ops, Bn)
    for rep in range(2):
        B.rwkvq_step_run(plan)
        torch.cuda.synchronize()
        assert B.rwkvq_device_status() == 0
        _check(ops, Bn)


def test_step_agrees_with_single_product_calls():
    ops = _build_ops(512, 1280, 1, 8, 6, seed=5)
    plan = _plan(ops, 8)
    B.rwkvq_step_run(plan)
    torch.cuda.synchronize()
    for e in ops:
        y1 = H.run_gemv(e["W"], e["mu"], e["x16"], e["xp16"])
        _, tol = H.reference(e["W"], e["mu"], e["x16"], e["xp16"])
        assert (np.abs(e["y"].double().cpu().numpy() - y1) <= tol).all()


def test_step_rejects_bad_plans():
    ops = _build_ops(512, 1280, 1, 1, 6, seed=6)
    plan = _plan(ops, 1)
    with pytest.raises(B.RwkvqError):
        B.rwkvq_step_run(plan[256:])         # not the buffer a plan was written to
    arr = B.make_ops([dict(desc=e["W"].desc, W=e["W"].dev, mu_desc=None, mu=None, x=e["xd"], xprev=None,
                           y=e["y"].half(), stage=e["stage"]) for e in ops[:1]])
    assert B.rwkvq_step_plan_bytes(arr, 1) == 0   # fp16 outputs are not supported by the step launch


@pytest.mark.parametrize("Bn,layout", [(4, "packed"), (4, "spread"), (16, "spread"), (1, "spread"), (8, "reversed")])
def test_step_run_host_matches_oracle(Bn, layout):
    """rwkvq_step_run_host (the call behind the benchmark's end-to-end figure): activations come from
    pinned host memory, results go back to pinned host memory, compared with the oracle there.
    "packed": small arenas, the copies run before and after the step.  "spread": the same products
    3 MB apart in arenas of tens of MB, so that the activations arrive in several chunks while the step
    runs and the outputs leave in several groups behind their stage barriers.  "reversed": outputs laid
    out against the order of the stages, which the call must answer with one copy at the end."""
    ops = _build_ops(512, 1280, 2, Bn, 6, seed=91 + Bn)
    # one arena for the activations and one for the outputs, as the stack runner lays them out
    gap = 0 if layout == "packed" else 3 << 20
    def al(n):
        return (n + 255) // 256 * 256 + gap
    act_off, y_off, slots = 0, 0, []
    for e in ops:
        xo = act_off; act_off += al(e["x16"].nbytes)
        po = None
        if e["mu"] is not None:
            po = act_off; act_off += al(e["xp16"].nbytes)
        slots.append([xo, po, y_off]); y_off += al(Bn * e["W"].oc * 4)
    if layout == "reversed":
        for sl, e in zip(slots, ops):
            sl[2] = y_off - sl[2] - al(Bn * e["W"].oc * 4)
    act_host = torch.zeros(act_off, dtype=torch.uint8).pin_memory()
    y_host = torch.zeros(y_off, dtype=torch.uint8).pin_memory()
    act_dev = torch.zeros(act_off, dtype=torch.uint8, device="cuda")
    y_dev = torch.full((y_off // 4,), float("nan"), dtype=torch.float32, device="cuda").view(torch.uint8)
    an = act_host.numpy()
    for e, (xo, po, yo) in zip(ops, slots):
        an[xo:xo + e["x16"].nbytes] = e["x16"].reshape(-1).view(np.uint8)
        e["xd"] = act_dev[xo:xo + e["x16"].nbytes].view(torch.float16).view(Bn, -1)
        if po is not None:
            an[po:po + e["xp16"].nbytes] = e["xp16"].reshape(-1).view(np.uint8)
            e["xpd"] = act_dev[po:po + e["xp16"].nbytes].view(torch.float16).view(Bn, -1)
        e["y"] = y_dev[yo:yo + Bn * e["W"].oc * 4].view(torch.float32).view(Bn, e["W"].oc)
    plan = _plan(ops, Bn)
    for rep in range(2):
        y_host.zero_()
        B.rwkvq_step_run_host(plan, act_host, act_dev, y_dev, y_host)
        torch.cuda.synchronize()
        assert B.rwkvq_device_status() == 0
        assert torch.equal(act_dev.cpu(), act_host)                      # the inputs went through the call
        yn = y_host.numpy()
        for e, (xo, po, yo) in zip(ops, slots):
            y = yn[yo:yo + Bn * e["W"].oc * 4].view(np.float32).reshape(Bn, -1).astype(np.float64)
            ref, tol = H.reference(e["W"], e["mu"], e["x16"], e["xp16"])
            assert np.isfinite(y).all() and (np.abs(y - ref) <= tol).all()
    B.rwkvq_step_plan_release(plan)
    with pytest.raises(B.RwkvqError):
        B.rwkvq_step_run(plan)                                           # the record of the plan is gone


def test_bounded_waits_run_out_and_the_plan_recovers():
    """No wait inside the step kernel is unbounded.  With a barrier target that can never be met
    (wait_skew) and a small poll limit every CTA gives up at its first stage barrier, the kernel
    returns, the status word says ETIMEOUT; after the status has been read the next run clears the
    barrier counters and matches the oracle again.  Nothing traps, faults or hangs."""
    for Bn in (1, 8):
        ops = _build_ops(512, 1280, 2, Bn, 6, seed=40 + Bn)
        plan = _plan(ops, Bn)
        B.rwkvq_step_run(plan)
        torch.cuda.synchronize()
        assert B.rwkvq_device_status() == 0
        _check(ops, Bn)
        B.rwkvq_step_set_wait(plan, poll_limit=2000, wait_skew=1)
        B.rwkvq_step_run(plan)
        torch.cuda.synchronize()                                         # the kernel returns by itself
        assert B.rwkvq_device_status() == 8                              # RWKVQ_ETIMEOUT, and the word is cleared
        assert B.rwkvq_device_status() == 0
        B.rwkvq_step_set_wait(plan, poll_limit=0, wait_skew=0)           # defaults again
        for rep in range(2):
            for e in ops:
                e["y"].fill_(float("nan"))
            B.rwkvq_step_run(plan)
            torch.cuda.synchronize()
            assert B.rwkvq_device_status() == 0
            _check(ops, Bn)


@pytest.mark.parametrize("Bn", [1, 8, 16])
def test_step_output_rows_end_inside_a_unit(Bn):
    """Row counts that end inside a 256-row unit (272 = one unit and one record) and inside a 128-row chunk
    (144): the 16-byte reductions of the flush stop at the last row; nothing beyond the outputs is written.
    An output that does not start on a 16-byte boundary is refused by the plan."""
    ops = []
    for k, (oc, ic) in enumerate([(272, 384), (144, 640), (256, 512), (272, 384)]):
        W = H.pack_sq(H.random_sq_codes(900 + 10 * Bn + k, oc, ic)) if k != 2 else H.pack_vq(H.random_vq_codes(900 + 10 * Bn + k, oc, ic, 6), 6)
        mu = H.pack_mu(H.random_mu_codes(950 + 10 * Bn + k, ic, 6), 6) if k % 2 == 0 else None
        x, xp = inputs.gen_activation_pair(990 + 10 * Bn + k, Bn, ic, n_outliers=4)
        x16, xp16 = x.astype(np.float16), xp.astype(np.float16)
        buf = torch.full((Bn * oc + 8,), float("nan"), dtype=torch.float32, device="cuda")
        y = buf[4:4 + Bn * oc].view(Bn, oc)
        ops.append(dict(W=W, mu=mu, x16=x16, xp16=xp16, stage=k // 2, xd=torch.from_numpy(x16).cuda(),
                        xpd=torch.from_numpy(xp16).cuda() if mu is not None else None, y=y, buf=buf))
    plan = _plan(ops, Bn)
    for _ in range(2):
        B.rwkvq_step_run(plan)
        torch.cuda.synchronize()
        assert B.rwkvq_device_status() == 0
        _check(ops, Bn)
    for e in ops:      # nothing outside the outputs was touched
        assert torch.isnan(e["buf"][:4]).all() and torch.isnan(e["buf"][4 + e["y"].numel():]).all()
    e = ops[0]
    bad = e["buf"][1:1 + Bn * e["W"].oc].view(Bn, e["W"].oc)
    arr = B.make_ops([dict(desc=e["W"].desc, W=e["W"].dev, mu_desc=e["mu"].desc, mu=e["mu"].dev, x=e["xd"], xprev=e["xpd"],
                           y=bad, stage=0)])
    assert B.rwkvq_step_plan_bytes(arr, Bn) == 0


@pytest.mark.parametrize("Bn", [5, 6, 10, 11])
def test_step_on_both_sides_of_the_stage_pre_pass(Bn):
    # 160 units on 148 SMs: two per CTA, 512 columns a row; 5 and 10 rows are mixed by the CTAs that read them, 6 and 11 by
    # the pre-pass (fewer items than warps on some CTAs, a half-empty last column tile, a product without a token shift)
    ops = []
    for k, (fmt, oc, ic, has_mu) in enumerate([("sq", 1024, 2432, True), ("vq6", 2048, 2560, True), ("sq", 1024, 2560, False)]):
        seed = 1000 + 10 * Bn + k
        W = H.pack_sq(H.random_sq_codes(seed, oc, ic)) if fmt == "sq" else H.pack_vq(H.random_vq_codes(seed, oc, ic, 6), 6)
        mu = H.pack_mu(H.random_mu_codes(seed + 3, ic, 6), 6) if has_mu else None
        x, xp = inputs.gen_activation_pair(seed + 6, Bn, ic, n_outliers=4)
        x16, xp16 = x.astype(np.float16), xp.astype(np.float16)
        ops.append(dict(W=W, mu=mu, x16=x16, xp16=xp16, stage=0, xd=torch.from_numpy(x16).cuda(),
                        xpd=torch.from_numpy(xp16).cuda() if has_mu else None,
                        y=torch.full((Bn, oc), float("nan"), dtype=torch.float32, device="cuda")))
    plan = _plan(ops, Bn)
    for rep in range(2):
        B.rwkvq_step_run(plan)
        torch.cuda.synchronize()
        assert B.rwkvq_device_status() == 0
        _check(ops, Bn)


class _HostArena:
    """The products' activations and outputs in one buffer each on the device and in page-locked memory, `gap` bytes apart."""

    def __init__(self, ops, Bn, gap):
        self.ops, self.Bn, self.slots, act, y = ops, Bn, [], 0, 0
        up = lambda n: (n + 255) // 256 * 256 + gap
        for e in ops:
            xo, po, yo = act, None, y
            act += up(e["x16"].nbytes)
            if e["mu"] is not None:
                po = act
                act += up(e["xp16"].nbytes)
            y += up(4 * Bn * e["W"].oc)
            self.slots.append((xo, po, yo))
        self.act_host, self.y_host = (torch.zeros(n, dtype=torch.uint8).pin_memory() for n in (act, y))
        self.act_dev = torch.zeros(act, dtype=torch.uint8, device="cuda")
        self.y_dev = torch.full((y // 4,), float("nan"), dtype=torch.float32, device="cuda").view(torch.uint8)
        for e, (xo, po, yo) in zip(ops, self.slots):
            e["xd"] = self.act_dev[xo:xo + e["x16"].nbytes].view(torch.float16).view(Bn, -1)
            if po is not None:
                e["xpd"] = self.act_dev[po:po + e["xp16"].nbytes].view(torch.float16).view(Bn, -1)
            e["y"] = self.y_dev[yo:yo + 4 * Bn * e["W"].oc].view(torch.float32).view(Bn, -1)
        self.fill(0)

    def fill(self, seed):
        """New activations in host memory; the outputs there are cleared."""
        an = self.act_host.numpy()
        for k, (e, (xo, po, _)) in enumerate(zip(self.ops, self.slots)):
            if seed:
                x, xp = inputs.gen_activation_pair(7000 + 100 * seed + k, self.Bn, e["W"].ic, n_outliers=4)
                e["x16"], e["xp16"] = x.astype(np.float16), xp.astype(np.float16)
            an[xo:xo + e["x16"].nbytes] = e["x16"].reshape(-1).view(np.uint8)
            if po is not None:
                an[po:po + e["xp16"].nbytes] = e["xp16"].reshape(-1).view(np.uint8)
        self.y_host.fill_(0xFF)

    def run(self, plan):
        B.rwkvq_step_run_host(plan, self.act_host, self.act_dev, self.y_dev, self.y_host)

    def check(self):
        yn = self.y_host.numpy()
        for e, (_, _, yo) in zip(self.ops, self.slots):
            y = yn[yo:yo + 4 * self.Bn * e["W"].oc].view(np.float32).reshape(self.Bn, -1).astype(np.float64)
            ref, tol = H.reference(e["W"], e["mu"], e["x16"], e["xp16"])
            assert np.isfinite(y).all() and (np.abs(y - ref) <= tol).all(), f"stage {e['stage']}"


@pytest.mark.parametrize("Bn", [4, 16])
def test_step_run_host_delivers_new_outputs_after_a_failed_wait(Bn):
    """A failed wait (here: another plan's) makes the next run of every plan clear its barrier counters, which hold many runs'
    arrivals.  The output copies wait for the arrivals of their own run, not for those: with new activations the host receives
    new outputs."""
    ops = _build_ops(512, 1280, 2, Bn, 6, seed=700 + Bn)
    arena = _HostArena(ops, Bn, 3 << 20)
    plan = _plan(ops, Bn)
    for _ in range(3):
        arena.run(plan)
    torch.cuda.synchronize()
    arena.check()
    other = _build_ops(256, 512, 1, 1, 6, seed=60)
    failing = _plan(other, 1)
    for seed in (1, 2):
        B.rwkvq_step_set_wait(failing, poll_limit=2000, wait_skew=1)
        B.rwkvq_step_run(failing)
        assert B.rwkvq_device_status() == 8
        arena.fill(seed)
        arena.run(plan)
        torch.cuda.synchronize()
        assert B.rwkvq_device_status() == 0
        arena.check()
        arena.run(plan)
        torch.cuda.synchronize()
        arena.check()


@pytest.mark.parametrize("Bn,gap", [(1, 24 << 10), (4, 24 << 10), (8, 50 << 10), (16, 0), (16, 100 << 10)])
def test_step_run_host_with_copies_of_half_a_megabyte_to_eight(Bn, gap):
    """Sizes from where the copies are overlapped on: first pieces of 256 KB and output groups of 128 KB, a few of each."""
    ops = _build_ops(512, 1280, 3, Bn, 6, seed=800 + Bn + gap)
    arena = _HostArena(ops, Bn, gap)
    total = arena.act_host.numel() + arena.y_host.numel()
    assert (512 << 10) <= total < (9 << 20)
    plan = _plan(ops, Bn)
    for seed in (0, 1, 2):
        arena.fill(seed)
        arena.run(plan)
        torch.cuda.synchronize()
        assert B.rwkvq_device_status() == 0
        arena.check()


def test_step_run_host_does_not_wait_for_another_streams_work():
    """Two streams: the first holds a second of other work in front of its step.  The step of the other does not occupy the SMs
    while its inputs wait behind that work: none of its (short) waits runs out."""
    arenas, plans = [], []
    for k in range(2):
        ops = _build_ops(512, 1280, 2, 4, 6, seed=900 + 50 * k)
        arenas.append(_HostArena(ops, 4, 64 << 10))
        plans.append(_plan(ops, 4))
        arenas[k].run(plans[k])
        torch.cuda.synchronize()
        arenas[k].check()
        arenas[k].fill(3 + k)
    busy, other = torch.cuda.Stream(), torch.cuda.Stream()
    B.rwkvq_step_set_wait(plans[1], poll_limit=20000)            # a wait for its inputs that lasts a second runs out
    with torch.cuda.stream(busy):
        torch.cuda._sleep(2_000_000_000)
        arenas[0].run(plans[0])
    with torch.cuda.stream(other):
        arenas[1].run(plans[1])
    other.synchronize()      # streams may share a hardware queue: how long this takes is not for a test
    assert B.rwkvq_device_status(other) == 0
    arenas[1].check()
    busy.synchronize()
    arenas[0].check()
    assert B.rwkvq_device_status() == 0
    for k in (0, 1, 1, 0):                                       # and the copy streams are used again
        arenas[k].fill(5 + k)
        arenas[k].run(plans[k])
        torch.cuda.synchronize()
        arenas[k].check()


@pytest.mark.parametrize("Bn", [1, 8, 16])
def test_captured_step_is_launched_many_times(Bn):
    """A step in a graph: its barriers hold in every launch of the graph and in runs between them."""
    ops = _build_ops(512, 1280, 2, Bn, 6, seed=1100 + Bn)
    plan = _plan(ops, Bn)
    B.rwkvq_step_run(plan)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        B.rwkvq_step_run(plan)
    for seed, launch in enumerate([graph.replay, graph.replay, lambda: B.rwkvq_step_run(plan), lambda: B.rwkvq_step_run(plan), graph.replay]):
        for k, e in enumerate(ops):
            x, xp = inputs.gen_activation_pair(9000 + 100 * seed + k, Bn, e["W"].ic, n_outliers=4)
            e["x16"], e["xp16"] = x.astype(np.float16), xp.astype(np.float16)
            e["xd"].copy_(torch.from_numpy(e["x16"]))
            if e["mu"] is not None:
                e["xpd"].copy_(torch.from_numpy(e["xp16"]))
            e["y"].fill_(float("nan"))
        launch()
        torch.cuda.synchronize()
        assert B.rwkvq_device_status() == 0
        _check(ops, Bn)


def test_captured_step_on_host_buffers():
    """The whole call in a graph, at a size that is overlapped outside one: every launch takes the host's present activations."""
    ops = _build_ops(512, 1280, 2, 4, 6, seed=1200)
    arena = _HostArena(ops, 4, 64 << 10)
    plan = _plan(ops, 4)
    arena.run(plan)
    torch.cuda.synchronize()
    arena.check()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        arena.run(plan)
    for seed, launch in enumerate([graph.replay, graph.replay, lambda: arena.run(plan), graph.replay]):
        arena.fill(10 + seed)
        launch()
        torch.cuda.synchronize()
        assert B.rwkvq_device_status() == 0
        arena.check()


@pytest.mark.parametrize("Bn", [2, 8, 11])
def test_step_with_many_products_in_one_stage(Bn):
    """Forty products that need not wait for one another (800 units, more inputs per CTA than it would mix itself): the CTAs' shares of
    the pre-pass begin and end inside products of both formats, with and without a token shift.  Resident inputs, and inputs
    that arrive from the host while the step runs."""
    ops = []
    for k in range(40):
        oc, ic = (1024, 1280) if k % 4 != 1 else (1008, 1152)
        seed = 1300 + 50 * Bn + k
        W = H.pack_vq(H.random_vq_codes(seed, oc, ic, 6), 6) if k % 4 == 0 else H.pack_sq(H.random_sq_codes(seed, oc, ic))
        mu = H.pack_mu(H.random_mu_codes(seed + 3, ic, 6), 6) if k % 3 else None
        x, xp = inputs.gen_activation_pair(seed + 6, Bn, ic, n_outliers=4)
        ops.append(dict(W=W, mu=mu, x16=x.astype(np.float16), xp16=xp.astype(np.float16), stage=0, xpd=None))
    arena = _HostArena(ops, Bn, 8 << 10)
    plan = _plan(ops, Bn)
    for seed in (0, 1):
        arena.fill(seed)
        arena.run(plan)
        torch.cuda.synchronize()
        assert B.rwkvq_device_status() == 0
        arena.check()
    for e in ops:
        e["y"].fill_(float("nan"))
    B.rwkvq_step_run(plan)
    torch.cuda.synchronize()
    assert B.rwkvq_device_status() == 0
    _check(ops, Bn)


@pytest.mark.parametrize("Bn,ic,bits", [(1, 2560, 3), (2, 2560, 8), (8, 2304, 6), (8, 2560, 3), (8, 2560, 8), (9, 2048, 3), (16, 1792, 8), (16, 2048, 3),
                                        (16, 2048, 6), (16, 4096, 8)])
def test_step_inputs_of_one_buffer_and_of_more(Bn, ic, bits):
    """A row of tiles a CTA: its columns fill an input buffer or go on in the next.  Inputs and decoded weights are exact, so that only the
    fp32 sums differ (1e-5 of |w| |x|)."""
    oc, g = 256 * 150, torch.Generator(device="cuda").manual_seed(Bn * ic + bits)
    desc = B.rwkvq_desc_for(oc, ic, B.RWKVQ_SQ if bits == 3 else B.RWKVQ_VQ, bits)
    w = (torch.randn((oc, ic), generator=g, device="cuda") * 0.02).half()
    image = torch.zeros(int(desc.image_bytes), dtype=torch.uint8, device="cuda")
    ws = torch.zeros(B.rwkvq_quantize_workspace_bytes(), dtype=torch.uint8, device="cuda")
    B.rwkvq_quantize_dev_async(w, oc, ic, desc.method, bits, image, ws, kmeans_iters=0, seed=1)
    x = torch.randn((Bn, ic), generator=g, device="cuda").half()
    y = torch.full((Bn, oc), float("nan"), device="cuda")
    ops = B.make_ops([dict(desc=desc, W=image, mu_desc=None, mu=None, x=x, xprev=None, y=y, stage=0)])
    plan = torch.zeros(B.rwkvq_step_plan_bytes(ops, Bn), dtype=torch.uint8, device="cuda")
    B.rwkvq_step_plan(ops, Bn, plan)
    B.rwkvq_step_run(plan)
    decoded = torch.empty((oc, ic), device="cuda")
    B.rwkvq_dequant(desc, image, decoded)
    ref = x.double() @ decoded.double().T
    bound = 1e-5 * x.double().norm(dim=1)[:, None] * decoded.double().norm(dim=1)[None]
    assert bool(((y.double() - ref).abs() <= bound).all())
    assert B.rwkvq_device_status() == 0
    B.rwkvq_step_plan_release(plan)


@pytest.mark.parametrize("kind", ["relu2", "gate", "plain"])
@pytest.mark.parametrize("Bn", [1, 3, 9])
def test_outputs_that_are_inputs_of_the_stage_before(kind, Bn):
    """Buffers in turn, y0 -> y1 -> y0: the outputs of the third stage are cleared only when all CTAs have read them as inputs of the second, whose
    matrix is a few units that most CTAs have no part in.  Against the same chain with a buffer for every output."""
    g = torch.Generator(device="cuda").manual_seed(Bn)
    ws = torch.zeros(B.rwkvq_quantize_workspace_bytes(), dtype=torch.uint8, device="cuda")

    def matrix(rows, cols):
        desc = B.rwkvq_desc_for(rows, cols, B.RWKVQ_SQ, 3)
        image = torch.zeros(int(desc.image_bytes), dtype=torch.uint8, device="cuda")
        B.rwkvq_quantize_dev_async((torch.randn((rows, cols), generator=g, device="cuda") * 0.05).half(), rows, cols, B.RWKVQ_SQ, 3, image, ws)
        return dict(desc=desc, W=image, mu_desc=None, mu=None, xprev=None)

    def zeros(cols):
        return torch.zeros((Bn, cols), device="cuda")

    w0, w1, w2, wg = matrix(1280, 1024), matrix(256, 1280), matrix(1280, 256), matrix(1280, 1024)
    x, x1 = torch.randn((Bn, 1024), generator=g, device="cuda").half(), torch.randn((Bn, 1280), generator=g, device="cuda").half()

    def chain(apart):
        y0, y1, gate = zeros(1280), zeros(256), zeros(1280)
        y2 = zeros(1280) if apart or kind == "plain" else gate if kind == "gate" else y0
        x1d = x1.clone() if apart else y2.view(torch.float16).view(-1)[:Bn * 1280].view(Bn, 1280)
        second = dict(x=x1d) if kind == "plain" else dict(x=None, **{"in": dict(kind=B.RWKVQ_IN_F32, src=y0, gate=gate) if kind == "gate" else
                                                                     dict(kind=B.RWKVQ_IN_RELU2, src=y0)})
        third = dict(x=x1[:, :256].contiguous()) if kind == "plain" else dict(x=None, **{"in": dict(kind=B.RWKVQ_IN_RELU2, src=y1)})
        keep = [dict(w0, x=x, y=y0, stage=0)] + ([dict(wg, x=x, y=gate, stage=0)] if kind == "gate" else [])
        keep += [dict(w1, y=y1, stage=1, **second), dict(w2, y=y2, stage=2, **third)]
        ops = B.make_ops(keep)
        plan = torch.zeros(B.rwkvq_step_plan_bytes(ops, Bn), dtype=torch.uint8, device="cuda")
        B.rwkvq_step_plan(ops, Bn, plan)
        out = []
        for _ in range(3 if apart else 60):
            if kind == "plain" and not apart:
                x1d.copy_(x1)
            B.rwkvq_step_run(plan)
            out.append((y1.clone(), y2.clone()))
        torch.cuda.synchronize()
        assert B.rwkvq_device_status() == 0
        B.rwkvq_step_plan_release(plan)
        return out

    want = chain(True)[0]
    assert all(bool((w != 0).any()) for w in want)
    for got in chain(False):
        for a, b in zip(got, want):      # sums in another order; an input may round to the other fp16 number (2^-11)
            assert float((a.double() - b.double()).norm()) <= 1e-3 * float(b.double().norm())


@pytest.mark.parametrize("Bn,bits", [(1, 3), (1, 6), (2, 8), (3, 6), (8, 3), (8, 8)])
@pytest.mark.parametrize("rows", [(16, 32, 37, 32), (16, 37, 48), (80, 75, 96, 80)])
def test_units_unpacked_ahead_of_their_inputs(rows, Bn, bits):
    """Stages of one to six units a CTA (rows of nine tiles on 148 SMs): plans of small stages (the first, of two units on average) unpack a group's first unit
    of a stage while its inputs are on their way, and go on to the next as before; plans of larger ones do not, and with one row the largest stages' first inputs are announced
    ahead of the rest.  Scalar rows end in half a unit.  Inputs and decoded weights are exact, so that only the fp32 sums differ (1e-5 of |w| |x|)."""
    ic, g = 2304, torch.Generator(device="cuda").manual_seed(10 * Bn + bits)
    ws = torch.zeros(B.rwkvq_quantize_workspace_bytes(), dtype=torch.uint8, device="cuda")
    keep = []
    for stage, r in enumerate(rows):
        oc = 256 * r - (112 if bits == 3 else 0)
        desc = B.rwkvq_desc_for(oc, ic, B.RWKVQ_SQ if bits == 3 else B.RWKVQ_VQ, bits)
        image = torch.zeros(int(desc.image_bytes), dtype=torch.uint8, device="cuda")
        w = (torch.randn((oc, ic), generator=g, device="cuda") * 0.02).half()
        B.rwkvq_quantize_dev_async(w, oc, ic, desc.method, bits, image, ws, kmeans_iters=0, seed=1)
        keep.append(dict(desc=desc, W=image, mu_desc=None, mu=None, x=torch.randn((Bn, ic), generator=g, device="cuda").half(), xprev=None,
                         y=torch.full((Bn, oc), float("nan"), device="cuda"), stage=stage))
    ops = B.make_ops(keep)
    forms = _forms(ops, Bn)
    assert forms.unpacked_ahead == (len(rows) == 4 and rows[0] == 16) and (forms.announced_heads > 0) == (rows[0] == 80 and Bn == 1)
    plan = torch.zeros(B.rwkvq_step_plan_bytes(ops, Bn), dtype=torch.uint8, device="cuda")
    B.rwkvq_step_plan(ops, Bn, plan)
    for _ in range(2):
        B.rwkvq_step_run(plan)
    for e in keep:
        decoded = torch.empty((e["desc"].oc, ic), device="cuda")
        B.rwkvq_dequant(e["desc"], e["W"], decoded)
        x = e["x"].double()
        bound = 1e-5 * x.norm(dim=1)[:, None] * decoded.double().norm(dim=1)[None]
        assert bool(((e["y"].double() - x @ decoded.double().T).abs() <= bound).all()), e["stage"]
    assert B.rwkvq_device_status() == 0
    B.rwkvq_step_plan_release(plan)


class _Large:
    """Stages of one scalar product each, rows of `tiles` column tiles, with token shifts where `shift` says so.  The inputs are mixed as the step mixes them and the
    decoded weights are exact, so that only the fp32 sums differ (1e-5 of |w| |x|)."""

    def __init__(self, Bn, rows, shift=True, tiles=9):
        self.Bn, self.keep, ic = Bn, [], 256 * tiles
        g = torch.Generator(device="cuda").manual_seed(100 * Bn + len(rows))
        ws = torch.zeros(B.rwkvq_quantize_workspace_bytes(), dtype=torch.uint8, device="cuda")
        for stage, r in enumerate(rows):
            oc = 256 * r
            desc = B.rwkvq_desc_for(oc, ic, B.RWKVQ_SQ, 3)
            image = torch.zeros(int(desc.image_bytes), dtype=torch.uint8, device="cuda")
            B.rwkvq_quantize_dev_async((torch.randn((oc, ic), generator=g, device="cuda") * 0.02).half(), oc, ic, desc.method, 3, image, ws)
            decoded = torch.empty((oc, ic), device="cuda")
            B.rwkvq_dequant(desc, image, decoded)
            x, xp = (torch.randn((Bn, ic), generator=g, device="cuda").half() for _ in range(2))
            mu = H.pack_mu(H.random_mu_codes(1500 + stage, ic, 6), 6) if shift else None
            mixed = x.double()
            if shift:      # the difference is rounded to fp32, then one fused multiply-add
                mixed = ((xp.float() - x.float()).double() * torch.from_numpy(mu.w_hat).cuda().double() + x.double()).float().half().double()
            self.keep.append((dict(desc=desc, W=image, mu_desc=mu.desc if shift else None, mu=mu.dev if shift else None, x=x, xprev=xp if shift else None,
                                   y=torch.zeros((Bn, oc), device="cuda"), stage=stage), decoded.double(), mixed, mu))
        self.ops = B.make_ops([e for e, *_ in self.keep])
        self.forms = _forms(self.ops, Bn)
        self.plan = torch.zeros(B.rwkvq_step_plan_bytes(self.ops, Bn), dtype=torch.uint8, device="cuda")
        B.rwkvq_step_plan(self.ops, Bn, self.plan)

    def run_and_check(self):
        for e, *_ in self.keep:
            e["y"].fill_(float("nan"))
        B.rwkvq_step_run(self.plan)
        assert B.rwkvq_device_status() == 0
        for e, w, x, _ in self.keep:
            bound = 1e-5 * x.norm(dim=1)[:, None] * w.norm(dim=1)[None]
            assert bool(((e["y"].double() - x @ w.T).abs() <= bound).all()), e["stage"]


@pytest.mark.parametrize("rows", [(80, 75, 96, 80, 77, 80, 91), (170, 60, 160)])
@pytest.mark.parametrize("shift", [True, False])
def test_announced_heads_of_one_row(rows, shift):
    """One row, large stages: the first tiles of a stage's first segment are announced ahead of the rest, with the previous token's row and mu_hat where
    there is a token shift.  In seven stages of one segment either buffer's announcements come to a third phase."""
    large = _Large(1, rows, shift)
    assert large.forms.pre_pass == 0 and large.forms.unpacked_ahead == 0 and large.forms.announced_heads > 0
    assert len(rows) < 7 or large.forms.most_heads >= 6
    for _ in range(3):
        large.run_and_check()
    B.rwkvq_step_plan_release(large.plan)


@pytest.mark.parametrize("Bn,rows,pre_pass", [(1, (80, 75, 96), 0), (2, (48, 45, 50), 0), (8, (48, 45, 50), 1)])
def test_bounded_waits_of_large_stages_run_out_and_the_plan_recovers(Bn, rows, pre_pass):
    """As test_bounded_waits_run_out_and_the_plan_recovers, for plans that do not unpack units ahead; with one row consumers wait for announced heads that
    never come."""
    large = _Large(Bn, rows)
    assert large.forms.pre_pass == pre_pass and large.forms.unpacked_ahead == 0 and (large.forms.announced_heads > 0) == (Bn == 1)
    large.run_and_check()
    B.rwkvq_step_set_wait(large.plan, poll_limit=2000, wait_skew=1)
    B.rwkvq_step_run(large.plan)
    torch.cuda.synchronize()                                         # the kernel returns by itself
    assert B.rwkvq_device_status() == 8                              # RWKVQ_ETIMEOUT, and the word is cleared
    assert B.rwkvq_device_status() == 0
    B.rwkvq_step_set_wait(large.plan, poll_limit=0, wait_skew=0)     # defaults again
    for _ in range(2):
        large.run_and_check()
    B.rwkvq_step_plan_release(large.plan)
