"""GPU parity of the element-wise operators between the projections of an RWKV block (Appendix A.1 Eq. 23 WKV,
Eq. 24 sigmoid gate, Eq. 27 squared ReLU and output gate), fused into the input stage of the persistent decode
step: a two-layer block chain is run for several tokens and every product, every recurrence state and every
previous-token state is checked against the oracle, each from the GPU's own upstream values (so an error
cannot hide behind the one before it)."""
import numpy as np
import pytest
import torch

from oracle import rwkvq_oracle as orc
from paper_2505_03803_b200 import binding as B
from paper_2505_03803_b200 import inputs

pytestmark = pytest.mark.gpu


class _Mat:
    def __init__(self, seed, oc, ic, method, std):
        w = (np.random.default_rng(seed).standard_normal((oc, ic)) * std).astype(np.float16)
        bits = 3 if method == B.RWKVQ_SQ else 6
        blob = B.rwkvq_pack(w, oc, ic, method, bits, kmeans_iters=2, seed=seed)
        c = blob.export_codes()
        self.w_hat = orc.sq_decode(c["q"], c["scale"], c["zero"]) if method == B.RWKVQ_SQ else orc.vq_decode(c["codebook"], c["q"])
        self.desc, self.dev, self.oc, self.ic = blob.desc, blob.to_device(), oc, ic


class _Mu:
    def __init__(self, seed, ic):
        blob = B.rwkvq_pack(inputs.gen_mu(seed, ic).reshape(1, -1), 1, ic, B.RWKVQ_VQ, 6, seed=seed)
        c = blob.export_codes()
        self.mu_hat = orc.mu_decode(c["codebook"], c["q"])
        self.desc, self.dev = blob.desc, blob.to_device()


def _f16(a):
    return np.asarray(a, dtype=np.float64).astype(np.float16).astype(np.float64)


def _build(d, h, layers, Bn, seed):
    """Ops of `layers` blocks: per block R, K, V (stage 0), O (1), cm_k and cm_r (2), cm_v (3)."""
    dev = "cuda"
    z32 = lambda *s: torch.zeros(s, dtype=torch.float32, device=dev)
    z16 = lambda *s: torch.zeros(s, dtype=torch.float16, device=dev)
    rng = np.random.default_rng(seed)
    x0 = z16(Bn, d)
    ops, entries = [], []
    prev = None           # (y_cm_r, y_cm_v) of the block before
    for l in range(layers):
        s0 = seed * 100 + l * 10
        m = {"R": _Mat(s0 + 1, d, d, B.RWKVQ_SQ, 0.08), "K": _Mat(s0 + 2, d, d, B.RWKVQ_VQ, 0.08),
             "V": _Mat(s0 + 3, d, d, B.RWKVQ_SQ, 0.08), "O": _Mat(s0 + 4, d, d, B.RWKVQ_SQ, 0.08),
             "cK": _Mat(s0 + 5, h, d, B.RWKVQ_SQ, 0.08), "cR": _Mat(s0 + 6, d, d, B.RWKVQ_SQ, 0.08),
             "cV": _Mat(s0 + 7, d, h, B.RWKVQ_VQ if l == 0 else B.RWKVQ_SQ, 0.08)}
        mu = {n: _Mu(s0 + 20 + i, d) for i, n in enumerate(("R", "K", "V", "cK", "cR"))}
        y = {n: z32(Bn, m[n].oc) for n in m}
        xs = {n: z16(Bn, d) for n in mu}                      # previous-token input, one per product
        st = {"a": z32(Bn, d), "b": z32(Bn, d), "p": torch.full((Bn, d), -1e30, dtype=torch.float32, device=dev),
              "u": torch.from_numpy((rng.standard_normal(d) * 0.3).astype(np.float32)).to(dev),
              "w": torch.from_numpy(rng.uniform(0.05, 1.0, d).astype(np.float32)).to(dev),
              "gain": torch.full((1,), 0.5 + 0.25 * l, dtype=torch.float32, device=dev)}
        blk = dict(m=m, mu=mu, y=y, xs=xs, st=st, prev=prev)
        for n in ("R", "K", "V"):
            if prev is None:
                xin = dict(kind=B.RWKVQ_IN_BUFFER, xprev_out=xs[n])
                e = dict(x=x0)
            else:
                xin = dict(kind=B.RWKVQ_IN_F32, src=prev[1], gate=prev[0], xprev_out=xs[n], rmsnorm=True)
                e = dict(x=None)
            e.update(desc=m[n].desc, W=m[n].dev, mu_desc=mu[n].desc, mu=mu[n].dev, xprev=xs[n], y=y[n], stage=4 * l, **{"in": xin})
            entries.append(e)
        entries.append(dict(desc=m["O"].desc, W=m["O"].dev, x=None, y=y["O"], stage=4 * l + 1,
                            **{"in": dict(kind=B.RWKVQ_IN_WKV, src=y["R"], k=y["K"], v=y["V"], state_a=st["a"], state_b=st["b"],
                                          state_p=st["p"], u=st["u"], w=st["w"], scale=st["gain"])}))
        for n in ("cK", "cR"):
            entries.append(dict(desc=m[n].desc, W=m[n].dev, mu_desc=mu[n].desc, mu=mu[n].dev, x=None, xprev=xs[n], y=y[n],
                                stage=4 * l + 2, **{"in": dict(kind=B.RWKVQ_IN_F32, src=y["O"], xprev_out=xs[n], rmsnorm=(n == "cK"))}))
        entries.append(dict(desc=m["cV"].desc, W=m["cV"].dev, x=None, y=y["cV"], stage=4 * l + 3,
                            **{"in": dict(kind=B.RWKVQ_IN_RELU2, src=y["cK"])}))
        prev = (y["cR"], y["cV"])
        ops.append(blk)
    return x0, ops, entries


def _np(t):
    return t.detach().double().cpu().numpy()


def _check_product(name, mat, x_ref, y_dev):
    ref, tol = orc.gemv(mat.w_hat, x_ref), orc.tolerance(mat.w_hat, x_ref)
    got = _np(y_dev)
    assert np.isfinite(got).all(), name
    err = np.abs(got - ref)
    assert (err <= tol + 1e-30).all(), f"{name}: max err/tol {float((err / np.maximum(tol, 1e-300)).max())}"


@pytest.mark.parametrize("Bn", [1, 3, 8, 16])
def test_block_chain_matches_oracle_token_by_token(Bn):
    d, h, layers = 256, 512, 2
    x0, blocks, entries = _build(d, h, layers, Bn, seed=Bn)
    ops = B.make_ops(entries)
    plan = torch.zeros(B.rwkvq_step_plan_bytes(ops, Bn), dtype=torch.uint8, device="cuda")
    B.rwkvq_step_plan(ops, Bn, plan)
    for token in range(4):
        x_host = inputs.gen_activation(1000 + 17 * Bn + token, Bn, d, 4).astype(np.float16)
        x0.copy_(torch.from_numpy(x_host).cuda())
        # states before the step
        before = [dict(xs={n: _np(t) for n, t in blk["xs"].items()},
                       a=_np(blk["st"]["a"]), b=_np(blk["st"]["b"]), p=_np(blk["st"]["p"])) for blk in blocks]
        B.rwkvq_step_run(plan)
        torch.cuda.synchronize()
        assert B.rwkvq_device_status() == 0
        for l, blk in enumerate(blocks):
            m, mu, y, st, bf = blk["m"], blk["mu"], blk["y"], blk["st"], before[l]
            # input of the time-mix projections: the token itself, or the gated output of the block before (Eq. 27)
            if blk["prev"] is None:
                x_t = x_host.astype(np.float64)
            else:
                x_t = _f16(orc.rms_normalize(orc.channel_mix_gate(_np(blk["prev"][0]), _np(blk["prev"][1]))))
            for n in ("R", "K", "V"):
                _check_product(f"token {token} layer {l} {n}", m[n], orc.token_shift(x_t, bf["xs"][n], mu[n].mu_hat), y[n])
                got_state = _np(blk["xs"][n])
                assert (np.abs(got_state - x_t) <= 2.0 ** -10 * np.abs(x_t) + 1e-7).all()    # within one fp16 step of x_t
            # Eq. 23 from the history sums before the step (stored scaled by e^{-p}), Eq. 24 gate
            a_true, b_true = bf["a"] * np.exp(bf["p"]), bf["b"] * np.exp(bf["p"])
            u, w = _np(st["u"]), _np(st["w"])
            wkv, a_new, b_new = orc.wkv_step(a_true, b_true, _np(y["K"]), _np(y["V"]), u, w)
            gain = float(st["gain"][0])
            _check_product(f"token {token} layer {l} O", m["O"], _f16(gain * orc.time_mix_gate(_np(y["R"]), wkv)), y["O"])
            ga, gb = _np(st["a"]) * np.exp(_np(st["p"])), _np(st["b"]) * np.exp(_np(st["p"]))
            # fp32 recurrence: relative to the magnitudes that are added (the numerator sum can cancel)
            a_scale = np.exp(-w) * np.abs(a_true) + np.exp(_np(y["K"])) * np.abs(_np(y["V"]))
            assert (np.abs(ga - a_new) <= 2e-5 * a_scale + 1e-30).all() and np.allclose(gb, b_new, rtol=2e-5, atol=1e-30)
            for n in ("cK", "cR"):       # cm_k reads the normalised output of time mixing, cm_r the plain one
                x_c = _f16(orc.rms_normalize(_np(y["O"]))) if n == "cK" else _f16(_np(y["O"]))
                _check_product(f"token {token} layer {l} {n}", m[n], orc.token_shift(x_c, bf["xs"][n], mu[n].mu_hat), y[n])
                assert (np.abs(_np(blk["xs"][n]) - x_c) <= 2.0 ** -10 * np.abs(x_c) + 1e-7).all()
            _check_product(f"token {token} layer {l} cV", m["cV"], _f16(orc.relu_squared(_np(y["cK"]))), y["cV"])
    B.rwkvq_step_plan_release(plan)


def test_block_first_token_and_argument_checks():
    # first token of a sequence: the history is empty, so wkv = v and the output projection sees sigmoid(r) * v
    Bn, d, h = 2, 256, 512
    x0, blocks, entries = _build(d, h, 1, Bn, seed=77)
    ops = B.make_ops(entries)
    plan = torch.zeros(B.rwkvq_step_plan_bytes(ops, Bn), dtype=torch.uint8, device="cuda")
    B.rwkvq_step_plan(ops, Bn, plan)
    x0.copy_(torch.from_numpy(inputs.gen_activation(5, Bn, d, 4).astype(np.float16)).cuda())
    B.rwkvq_step_run(plan)
    torch.cuda.synchronize()
    blk = blocks[0]
    y = blk["y"]
    _check_product("first token O", blk["m"]["O"], _f16(0.5 * orc.sigmoid(_np(y["R"])) * _np(y["V"])), y["O"])
    B.rwkvq_step_plan_release(plan)
    # a WKV input without its state, and an unknown kind, are refused before anything is planned
    bad = [dict(e) for e in entries]
    bad[3] = dict(bad[3], **{"in": dict(kind=B.RWKVQ_IN_WKV, src=y["R"], k=y["K"], v=y["V"])})
    assert B.rwkvq_step_plan_bytes(B.make_ops(bad), Bn) == 0
    bad = [dict(e) for e in entries]
    bad[6] = dict(bad[6], **{"in": dict(kind=9, src=y["cK"])})
    assert B.rwkvq_step_plan_bytes(B.make_ops(bad), Bn) == 0


def _decode(st, op):
    codes, mu_codes = st.host_codes(op)
    w_hat = orc.sq_decode(codes["q"], codes["scale"], codes["zero"]) if op.method == B.RWKVQ_SQ else orc.vq_decode(codes["codebook"], codes["q"])
    mu_hat = orc.mu_decode(mu_codes["codebook"], mu_codes["q"]) if mu_codes is not None else None
    return w_hat, mu_hat


@pytest.mark.parametrize("batch", [1, 16])
def test_chained_blocks_at_7b_width_sampled(batch):
    """The chain bench.py times (BlockStack), two blocks of the 7B-class width: after two tokens, one product of
    every kind of input operator is recomputed by the oracle from the values the GPU holds upstream."""
    from paper_2505_03803_b200 import stack as stack_mod
    st = stack_mod.BlockStack(4096, 14336, 2, 64, batch, n_outliers=8, tag="c3_7b", kmeans_iters=2)
    by = {(o.layer, o.name): o for o in st.ops}
    for token in range(2):
        st.set_token(50 + token)
        prev_R1 = _np(by[(1, "R")].xprev)
        prev_ck0 = _np(by[(0, "cm_k")].xprev)
        a0, b0, p0 = (_np(st.states[0][k]) for k in ("a", "b", "p"))
        st.run_step_host()
        torch.cuda.synchronize()
        assert B.rwkvq_device_status() == 0
    y = {k: _np(o.y) for k, o in by.items()}
    assert all(np.isfinite(v).all() for v in y.values())
    # block 1, R: gated and normalised output of block 0 (Eq. 27), token-shift mix with the token before
    w_hat, mu_hat = _decode(st, by[(1, "R")])
    x_t = _f16(orc.rms_normalize(orc.channel_mix_gate(y[(0, "cm_r")], y[(0, "cm_v")])))
    _check_product("block 1 R", type("M", (), {"w_hat": w_hat}), orc.token_shift(x_t, prev_R1, mu_hat), by[(1, "R")].y)
    # block 0, O: WKV (Eq. 23) from the history before the second token, sigmoid gate (Eq. 24)
    w_hat, _ = _decode(st, by[(0, "O")])
    wkv, _, _ = orc.wkv_step(a0 * np.exp(p0), b0 * np.exp(p0), y[(0, "K")], y[(0, "V")], _np(st.states[0]["u"]), _np(st.states[0]["w"]))
    _check_product("block 0 O", type("M", (), {"w_hat": w_hat}), _f16(orc.time_mix_gate(y[(0, "R")], wkv)), by[(0, "O")].y)
    # block 0, cm_k: normalised output of time mixing with its own token shift; cm_v: squared ReLU (Eq. 27)
    w_hat, mu_hat = _decode(st, by[(0, "cm_k")])
    x_c = _f16(orc.rms_normalize(y[(0, "O")]))
    _check_product("block 0 cm_k", type("M", (), {"w_hat": w_hat}), orc.token_shift(x_c, prev_ck0, mu_hat), by[(0, "cm_k")].y)
    w_hat, _ = _decode(st, by[(1, "cm_v")])
    _check_product("block 1 cm_v", type("M", (), {"w_hat": w_hat}), _f16(orc.relu_squared(y[(1, "cm_k")])), by[(1, "cm_v")].y)


@pytest.mark.parametrize("exponents", [(0,), (1, 23, 24, 60), (99, 122, 123, 124, 125), (126,), (127,)])
def test_reciprocal_of_the_sigmoids_is_the_rounded_division(exponents):
    """The sigmoids' reciprocal against numpy's fp32 division, which IEEE rounds correctly: the same bits for every significand of
    the binades [2^e, 2^(e+1)), among them those whose reciprocal is subnormal (from 2^126 on), and at infinity."""
    frac = torch.arange(1 << 23, dtype=torch.int32, device="cuda")
    for e in exponents:
        y = (frac | ((e + 127) << 23)).view(torch.float32)
        out = torch.empty_like(y)
        B.rwkvq_step_reciprocal(y, out)
        want = np.float32(1.0) / y.cpu().numpy()
        assert np.array_equal(out.cpu().numpy().view(np.uint32), want.view(np.uint32)), e
    ends = torch.tensor([1.0, float("inf"), float("nan"), 3.4028234e38, 2.0 ** 126, 1e37], device="cuda")
    out = torch.empty_like(ends)
    B.rwkvq_step_reciprocal(ends, out)
    got = out.cpu().numpy()
    assert got[1] == 0.0 and np.isnan(got[2]) and np.array_equal(got[[0, 3, 4, 5]], np.float32(1.0) / ends.cpu().numpy()[[0, 3, 4, 5]])


@pytest.mark.parametrize("Bn,oc,bits", [(1, 256, 3), (3, 512, 6), (8, 384, 3), (8, 1024, 8), (9, 512, 6)])
def test_squared_inputs_of_one_stage(Bn, oc, bits):
    """y1 = W1 relu(y0)^2 of y0 = W0 x: squared by every CTA for itself up to eight rows, in the pre-pass above."""
    ic, g = 1024, torch.Generator(device="cuda").manual_seed(Bn + oc)
    ws = torch.zeros(B.rwkvq_quantize_workspace_bytes(), dtype=torch.uint8, device="cuda")

    def matrix(rows, cols, b):
        desc = B.rwkvq_desc_for(rows, cols, B.RWKVQ_SQ if b == 3 else B.RWKVQ_VQ, b)
        image = torch.zeros(int(desc.image_bytes), dtype=torch.uint8, device="cuda")
        B.rwkvq_quantize_dev_async((torch.randn((rows, cols), generator=g, device="cuda") * 0.02).half(), rows, cols, desc.method, b, image, ws, kmeans_iters=1, seed=1)
        decoded = torch.empty((rows, cols), device="cuda")
        B.rwkvq_dequant(desc, image, decoded)
        return desc, image, decoded.double()

    (d0, w0, m0), (d1, w1, m1) = matrix(1280, ic, 3), matrix(oc, 1280, bits)
    x = torch.randn((Bn, ic), generator=g, device="cuda").half()
    y0, y1 = torch.zeros((Bn, 1280), device="cuda"), torch.zeros((Bn, oc), device="cuda")
    ops = B.make_ops([dict(desc=d0, W=w0, mu_desc=None, mu=None, x=x, xprev=None, y=y0, stage=0),
                      dict(desc=d1, W=w1, mu_desc=None, mu=None, x=None, xprev=None, y=y1, stage=1, **{"in": dict(kind=B.RWKVQ_IN_RELU2, src=y0)})])
    plan = torch.zeros(B.rwkvq_step_plan_bytes(ops, Bn), dtype=torch.uint8, device="cuda")
    B.rwkvq_step_plan(ops, Bn, plan)
    for _ in range(20):
        B.rwkvq_step_run(plan)
    torch.cuda.synchronize()
    assert B.rwkvq_device_status() == 0
    k = y0.double()
    assert bool(((k - x.double() @ m0.T).abs() <= 2e-3 * x.double().norm(dim=1)[:, None] * m0.norm(dim=1)[None]).all())
    squares = k.clamp_min(0.0) ** 2
    assert bool(((y1.double() - squares @ m1.T).abs() <= 2e-3 * squares.norm(dim=1)[:, None] * m1.norm(dim=1)[None]).all())
    B.rwkvq_step_plan_release(plan)


@pytest.mark.parametrize("Bn,rows,kinds", [(1, 17, "pspspp"), (1, 70, "spspps"), (3, 33, "psppsspp"), (8, 17, "psppsspp"), (8, 16, "sspps"), (2, 64, "pspsp")])
def test_copied_inputs_behind_squared_ones(Bn, rows, kinds):
    """Stages of squared (s) and of plain (p) inputs by turns: the copies of a plain stage land where squares that the CTA stored itself lay before.  Every product
    has inputs of its own, squares rounded to fp16 as the step rounds them, so that only the fp32 sums differ (1e-5 of |w| |x|)."""
    ic, g = 2304, torch.Generator(device="cuda").manual_seed(Bn * rows)
    oc = 256 * rows
    ws = torch.zeros(B.rwkvq_quantize_workspace_bytes(), dtype=torch.uint8, device="cuda")
    desc = B.rwkvq_desc_for(oc, ic, B.RWKVQ_SQ, 3)
    image = torch.zeros(int(desc.image_bytes), dtype=torch.uint8, device="cuda")
    B.rwkvq_quantize_dev_async((torch.randn((oc, ic), generator=g, device="cuda") * 0.02).half(), oc, ic, desc.method, 3, image, ws)
    decoded = torch.empty((oc, ic), device="cuda")
    B.rwkvq_dequant(desc, image, decoded)
    keep, want = [], []
    for stage, kind in enumerate(kinds):
        x = torch.randn((Bn, ic), generator=g, device="cuda")
        e = dict(desc=desc, W=image, mu_desc=None, mu=None, xprev=None, y=torch.zeros((Bn, oc), device="cuda"), stage=stage)
        e.update(dict(x=None, **{"in": dict(kind=B.RWKVQ_IN_RELU2, src=x)}) if kind == "s" else dict(x=x.half()))
        keep.append((e, x))
        want.append((x.clamp_min(0.0).square() if kind == "s" else x).half().double())
    ops = B.make_ops([e for e, _ in keep])
    forms = B.rwkvq_step_plan_forms(ops, Bn, torch.cuda.get_device_properties(0).multi_processor_count)
    assert forms.squared > 0 and forms.behind_squared > 0
    plan = torch.zeros(B.rwkvq_step_plan_bytes(ops, Bn), dtype=torch.uint8, device="cuda")
    B.rwkvq_step_plan(ops, Bn, plan)
    for _ in range(10):
        B.rwkvq_step_run(plan)
        for (e, _), x in zip(keep, want):
            bound = 1e-5 * x.norm(dim=1)[:, None] * decoded.double().norm(dim=1)[None]
            assert bool(((e["y"].double() - x @ decoded.double().T).abs() <= bound).all()), e["stage"]
    assert B.rwkvq_device_status() == 0
    B.rwkvq_step_plan_release(plan)
