"""Device quantizers (rwkvq_quantize_dev, rwkvq_calib_representative) against the oracle.

SQ (Section 3.2 Eq. 2): codes, scales and zero points bit-exact, image payload identical to the host
packer's.  VQ (Eq. 3) and the weighted k-means of Section 4.2: codebook values have several correct
answers, so what is unique is compared exactly (the assignment given the codebook, zero error on few
distinct vectors) and the rest through the loss the method minimises, next to the oracle's own run.
"""
import numpy as np
import pytest
import torch

from oracle import rwkvq_oracle as orc
from paper_2505_03803_b200 import binding as B

pytestmark = pytest.mark.gpu


def quantize_dev(w16, method, bits, elem_weight=None, seed=0, iters=10):
    oc, ic = (1, w16.shape[0]) if w16.ndim == 1 else w16.shape
    d0 = B.rwkvq_desc_for(oc, ic, method, bits)
    wd = torch.from_numpy(np.ascontiguousarray(w16)).cuda()
    img = torch.full((int(d0.image_bytes),), 0xAB, dtype=torch.uint8, device="cuda")
    ws = torch.empty(B.rwkvq_quantize_workspace_bytes(), dtype=torch.uint8, device="cuda")
    ew = None if elem_weight is None else torch.from_numpy(np.ascontiguousarray(elem_weight, dtype=np.float32)).cuda()
    d = B.rwkvq_quantize_dev(wd, oc, ic, method, bits, img, ws, elem_weight=ew, kmeans_iters=iters, seed=seed)
    torch.cuda.synchronize()
    assert d.image_bytes == d0.image_bytes
    return d, img


def sq_cases():
    rng = np.random.default_rng(42)
    out = {}
    out["gauss_512"] = (rng.standard_normal((512, 512)) * 0.02).astype(np.float16)
    out["ragged_272x384"] = (rng.standard_normal((272, 384)) * 0.02).astype(np.float16)
    out["student_1024x768"] = (rng.standard_t(3, (1024, 768)) * 0.01).astype(np.float16)
    w = (rng.standard_normal((256, 1024)) * 0.02).astype(np.float16)
    w[0, :128] = 0.0                       # constant groups: zero, positive, negative
    w[1, :128] = 0.375
    w[2, 128:256] = -0.0625
    w[3, :128] = np.float16(6e-8)          # subnormal constant
    w[4, :128] = np.where(np.arange(128) % 2 == 0, np.float16(6e-8), np.float16(1.2e-7))   # scale underflows to 0
    w[5, :128] = (100.0 + rng.uniform(0, 0.5, 128)).astype(np.float16)                      # far from zero: z saturates
    w[6, :128] = (np.arange(128) % 15) * 0.5                                                # s = 1: quotients on ties
    w[7, :128] = -((np.arange(128) % 15) * 0.5)
    w[8, :128] = (np.arange(128) % 8).astype(np.float16) * np.float16(0.1)                  # ramp: q = t
    w[9, :128] = rng.choice([-60000.0, 60000.0, 1e-4], 128)                                # full fp16 range
    w[10, 896:1024] = rng.uniform(-1, 1, 128) * 2.0 ** -14                                  # around the subnormal boundary
    out["special_256x1024"] = w
    return out


@pytest.mark.parametrize("name", list(sq_cases().keys()))
def test_sq_device_quantizer_is_bit_exact(name):
    w16 = sq_cases()[name]
    oc, ic = w16.shape
    d, img = quantize_dev(w16, B.RWKVQ_SQ, 3)
    host = img.cpu().numpy()
    d2, codes = B.rwkvq_image_unpack(host)
    q, s, z = orc.sq_encode(w16)
    assert (d2.oc, d2.ic, d2.method, d2.bits) == (oc, ic, B.RWKVQ_SQ, 3)
    assert np.array_equal(np.asarray(codes["q"]).reshape(oc, ic), q)
    assert np.array_equal(np.asarray(codes["scale"]).view(np.uint16).reshape(s.shape), s.view(np.uint16))
    # zero points are compared as numbers: a group whose minimum is 0 gets z = -0.0 from the oracle's
    # round(-min / s) and +0.0 from a clamp written with max(); both denote the same zero point
    assert np.array_equal(np.asarray(codes["zero"]).reshape(z.shape).astype(np.float64), z.astype(np.float64))
    # the whole payload (padding included) equals the host packer's
    ref = B.rwkvq_pack(w16, oc, ic, B.RWKVQ_SQ, 3).image()
    assert np.array_equal(host[256:], ref[256:])      # (both write +0.0 for such a zero point)


def test_sq_device_image_feeds_the_products():
    rng = np.random.default_rng(3)
    w16 = (rng.standard_normal((512, 768)) * 0.02).astype(np.float16)
    d, img = quantize_dev(w16, B.RWKVQ_SQ, 3)
    q, s, z = orc.sq_encode(w16)
    w_hat = orc.sq_decode(q, s, z)
    out = torch.empty((512, 768), dtype=torch.float32, device="cuda")
    B.rwkvq_dequant(d, img, out)
    assert np.array_equal(out.cpu().numpy().astype(np.float64), w_hat.astype(np.float32).astype(np.float64))
    x = rng.standard_normal((3, 768)).astype(np.float16)
    y = torch.empty((3, 512), dtype=torch.float32, device="cuda")
    ws = torch.zeros(max(256, B.rwkvq_gemv_workspace_bytes(d, 3)), dtype=torch.uint8, device="cuda")
    B.rwkvq_gemv(d, img, None, None, torch.from_numpy(x).cuda(), None, 3, y, ws)
    torch.cuda.synchronize()
    ref = orc.gemv(w_hat, x.astype(np.float64))
    tol = orc.tolerance(w_hat, x.astype(np.float64))
    assert np.all(np.abs(y.cpu().numpy().astype(np.float64) - ref) <= tol)


def test_sq_device_image_of_special_groups_feeds_the_products():
    # the matrix of degenerate groups (constants, +-0, the full fp16 range, subnormals): its device
    # image must decode to the oracle's values bit for bit and multiply within the tolerance
    w16 = sq_cases()["special_256x1024"]
    oc, ic = w16.shape
    d, img = quantize_dev(w16, B.RWKVQ_SQ, 3)
    q, s, z = orc.sq_encode(w16)
    w_hat = orc.sq_decode(q, s, z)
    out = torch.empty((oc, ic), dtype=torch.float32, device="cuda")
    B.rwkvq_dequant(d, img, out)
    assert np.array_equal(out.cpu().numpy().astype(np.float64), w_hat)
    rng = np.random.default_rng(12)
    for Bn in (1, 5):
        x = rng.standard_normal((Bn, ic)).astype(np.float16)
        y = torch.empty((Bn, oc), dtype=torch.float32, device="cuda")
        ws = torch.zeros(max(256, B.rwkvq_gemv_workspace_bytes(d, Bn)), dtype=torch.uint8, device="cuda")
        B.rwkvq_gemv(d, img, None, None, torch.from_numpy(x).cuda(), None, Bn, y, ws)
        torch.cuda.synchronize()
        ref = orc.gemv(w_hat, x.astype(np.float64))
        tol = orc.tolerance(w_hat, x.astype(np.float64))
        got = y.cpu().numpy().astype(np.float64)
        assert np.isfinite(got).all() and np.all(np.abs(got - ref) <= tol)


def tile_vectors(w16, tr, tc):
    return w16[tr * 256:(tr + 1) * 256, tc * 256:(tc + 1) * 256].astype(np.float64).reshape(-1, 2)


@pytest.mark.parametrize("bits,oc,ic", [(6, 512, 768), (8, 256, 512)])
def test_vq_device_quantizer_valid_and_as_good_as_the_oracle(bits, oc, ic):
    rng = np.random.default_rng(10 + bits)
    E = 1 << bits
    w16 = (rng.standard_t(3, (oc, ic)) * 0.01).astype(np.float16)
    d, img = quantize_dev(w16, B.RWKVQ_VQ, bits, seed=5)
    _, img_again = quantize_dev(w16, B.RWKVQ_VQ, bits, seed=5)
    assert torch.equal(img, img_again), "the device quantizer is not reproducible"
    _, codes = B.rwkvq_image_unpack(img.cpu().numpy())
    cbs = np.asarray(codes["codebook"]).reshape(oc // 256, ic // 256, E, 2)
    idx = np.asarray(codes["q"]).reshape(oc, ic // 2)
    assert np.isfinite(cbs.astype(np.float64)).all()
    cb_o, idx_o = orc.vq_encode(w16, entries=E, seed=5)
    mse_dev = mse_orc = 0.0
    for tr in range(oc // 256):
        for tc in range(ic // 256):
            v = tile_vectors(w16, tr, tc)
            c = cbs[tr, tc].astype(np.float64)
            ix = idx[tr * 256:(tr + 1) * 256, tc * 128:(tc + 1) * 128].reshape(-1)
            # unique given the codebook: nearest centre, lowest index on ties (Eq. 3)
            assert np.array_equal(ix, orc._nearest(v, c))
            mse_dev += float(((v - c[ix]) ** 2).sum())
            co = cb_o[tr, tc].astype(np.float64)
            io = idx_o[tr * 256:(tr + 1) * 256, tc * 128:(tc + 1) * 128].reshape(-1)
            mse_orc += float(((v - co[io]) ** 2).sum())
    assert mse_dev <= 1.10 * mse_orc, (mse_dev, mse_orc)
    # the image is what the products read
    out = torch.empty((oc, ic), dtype=torch.float32, device="cuda")
    B.rwkvq_dequant(d, img, out)
    assert np.array_equal(out.cpu().numpy().astype(np.float64), orc.vq_decode(cbs, idx))


def test_vq_device_lloyd_iterations_lower_the_loss():
    rng = np.random.default_rng(2)
    w16 = (rng.standard_normal((256, 256)) * 0.02).astype(np.float16)
    v = tile_vectors(w16, 0, 0)
    losses = []
    for iters in (0, 1, 3, 10):
        _, img = quantize_dev(w16, B.RWKVQ_VQ, 6, seed=9, iters=iters)
        _, codes = B.rwkvq_image_unpack(img.cpu().numpy())
        c = np.asarray(codes["codebook"]).reshape(64, 2).astype(np.float64)
        losses.append(float(((v - c[np.asarray(codes["q"]).reshape(-1)]) ** 2).sum()))
    assert losses[1] < losses[0] and losses[2] < losses[1] and losses[3] < losses[2]


@pytest.mark.parametrize("bits", [6, 8])
def test_vq_device_zero_error_on_few_distinct_vectors(bits):
    rng = np.random.default_rng(1)
    E = 1 << bits
    protos = (rng.standard_normal((E - 3, 2)) * 0.05).astype(np.float16)
    pick = rng.integers(0, len(protos), (256, 128))
    w16 = protos[pick].reshape(256, 256)
    _, img = quantize_dev(w16, B.RWKVQ_VQ, bits, seed=1)
    _, codes = B.rwkvq_image_unpack(img.cpu().numpy())
    w_hat = orc.vq_decode(np.asarray(codes["codebook"]).reshape(1, 1, E, 2), np.asarray(codes["q"]).reshape(256, 128))
    assert np.array_equal(w_hat, w16.astype(np.float64))
    const = np.full((256, 512), np.float16(-0.3125))
    _, img = quantize_dev(const, B.RWKVQ_VQ, bits)
    _, codes = B.rwkvq_image_unpack(img.cpu().numpy())
    w_hat = orc.vq_decode(np.asarray(codes["codebook"]).reshape(1, 2, E, 2), np.asarray(codes["q"]).reshape(256, 256))
    assert np.array_equal(w_hat, const.astype(np.float64))


def calib_samples(S, n, seed):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((S, n)) * (1.0 + 4.0 * (rng.random(n) < 0.05))[None, :] + rng.standard_normal(n)[None, :] * 0.5
    hot = rng.random((S, n)) < 0.01
    x[hot] *= 20.0
    return x.astype(np.float32)


@pytest.mark.parametrize("S,n,pct", [(128, 2048, 1.0), (128, 1000, 5.0), (101, 70, 10.0), (16, 33, 0.0), (7, 5, 25.0)])
def test_representative_activation_matches_oracle(S, n, pct):
    x = calib_samples(S, n, S + n)
    xd = torch.from_numpy(x).cuda()
    rep = torch.empty(n, dtype=torch.float32, device="cuda")
    rsq = torch.empty(n, dtype=torch.float32, device="cuda")
    B.rwkvq_calib_representative(xd, pct, rep, rsq)
    torch.cuda.synchronize()
    ref = orc.representative_activation(x.astype(np.float64), pct)
    got = rep.cpu().numpy().astype(np.float64)
    # fp64 mean in another summation order, then one rounding to fp32
    assert np.all(np.abs(got - ref) <= np.abs(ref) * 2.0 ** -23 + 1e-12)
    assert np.all(np.abs(rsq.cpu().numpy().astype(np.float64) - ref * ref) <= ref * ref * 2.0 ** -22 + 1e-12)


@pytest.mark.parametrize("ic,bits", [(2048, 6), (4096, 6), (5120, 8)])
def test_weighted_mu_quantizer(ic, bits):
    rng = np.random.default_rng(ic)
    E = 1 << bits
    mu16 = rng.uniform(0.0, 1.0, ic).astype(np.float16)
    x = calib_samples(128, ic, 7)
    rep = orc.representative_activation(x.astype(np.float64), 1.0)
    xd = torch.from_numpy(x).cuda()
    rsq = torch.empty(ic, dtype=torch.float32, device="cuda")
    B.rwkvq_calib_representative(xd, 1.0, None, rsq)
    torch.cuda.synchronize()
    wts = rsq.cpu().numpy()
    assert np.all(np.abs(wts.astype(np.float64) - rep * rep) <= rep * rep * 2.0 ** -22 + 1e-12)
    v = mu16.astype(np.float64).reshape(-1, 2)
    w2 = wts.astype(np.float64).reshape(-1, 2)

    def loss_of(img):
        _, codes = B.rwkvq_image_unpack(img.cpu().numpy())
        c = np.asarray(codes["codebook"]).reshape(E, 2).astype(np.float64)
        ix = np.asarray(codes["q"]).reshape(-1)
        return c, ix, float((w2 * (v - c[ix]) ** 2).sum())

    d, img = quantize_dev(mu16, B.RWKVQ_VQ, bits, elem_weight=wts, seed=3)
    c, ix, loss_w = loss_of(img)
    assert np.array_equal(ix, orc._nearest(v, c, w2))          # unique given the codebook (Eq. 19)
    loss_o = 0.0
    for sd in (3, 4, 5):      # the oracle's own spread over seeds is of the order of ten per cent
        cb_o, ix_o = orc.mu_encode(mu16, entries=E, seed=sd, act_sq=wts.astype(np.float64))
        loss_o += float((w2 * (v - cb_o.astype(np.float64)[ix_o]) ** 2).sum()) / 3.0
    assert loss_w <= 1.35 * loss_o, (loss_w, loss_o)
    # the plain codebook of the same vector is worse under Eq. 19
    _, img_plain = quantize_dev(mu16, B.RWKVQ_VQ, bits, seed=3)
    c_p, ix_p, loss_p = loss_of(img_plain)
    assert np.array_equal(ix_p, orc._nearest(v, c_p))
    assert loss_w < loss_p
    # the image decodes to the codebook entries
    out = torch.empty(ic, dtype=torch.float32, device="cuda")
    B.rwkvq_dequant(d, img, out)
    assert np.array_equal(out.cpu().numpy().astype(np.float64), orc.mu_decode(c.astype(np.float16), ix))


@pytest.mark.parametrize("ic,bits", [(128, 6), (2176, 6), (8192, 6), (8448, 6), (8448, 8)])
@pytest.mark.parametrize("weighted", [False, True])
def test_mu_quantizer_ties_zero_weights_and_sizes(ic, bits, weighted):
    """Sizes around the warps of the seeding, the shares of the assignment and the table of the sums; equal vectors,
    equal distances and weights of zero: the indices are the oracle's nearest entries, lowest first."""
    rng = np.random.default_rng(ic + bits)
    mu16 = (rng.integers(0, 24, ic) / 16.0).astype(np.float16)
    mu16[: ic // 2] += rng.uniform(0.0, 0.01, ic // 2).astype(np.float16)
    wts = None
    if weighted:
        wts = (rng.standard_normal(ic) ** 2).astype(np.float32)
        wts[rng.random(ic) < 0.1] = 0.0
        wts[:8] = 0.0
        wts[8:16] = 1e-38
    _, img = quantize_dev(mu16, B.RWKVQ_VQ, bits, elem_weight=wts, seed=5, iters=4)
    _, codes = B.rwkvq_image_unpack(img.cpu().numpy())
    c = np.asarray(codes["codebook"]).reshape(1 << bits, 2).astype(np.float64)
    w2 = None if wts is None else wts.astype(np.float64).reshape(-1, 2)
    want = orc._nearest(mu16.astype(np.float64).reshape(-1, 2), c, w2)
    assert np.array_equal(np.asarray(codes["q"]).reshape(-1), want)
    _, again = quantize_dev(mu16, B.RWKVQ_VQ, bits, elem_weight=wts, seed=5, iters=4)
    assert torch.equal(img, again)


def _drawn_seeds(v16, entries, seed):
    """k-means++ draws as the device defines them: fp32 distances summed over runs of 64 vectors in order, run sums by a scan over
    32 lanes and then warp by warp; a draw takes the last vector whose running sum begins at or below the target."""
    f32, mask, n = np.float32, (1 << 64) - 1, len(v16)

    def unit(k):
        z = (seed + (k + 1) * 0x9E3779B97F4A7C15) & mask
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        return ((z ^ (z >> 31)) >> 11) * 2.0 ** -53

    lanes = -(-n // 2048) * 32
    v = v16.astype(f32)
    dist = np.zeros(lanes * 64, f32)
    dist[:n] = np.inf
    at, picks = int(unit(0) * n) % n, []
    for e in range(entries):
        picks.append(at)
        if e + 1 == entries:
            return v16[picks]
        d = v - v[at]
        # one rounding of dx * dx + (dy * dy): exact enough in the long type
        dist[:n] = np.minimum(dist[:n], (d[:, 0].astype(np.longdouble) ** 2 + (d[:, 1] * d[:, 1]).astype(np.longdouble)).astype(f32))
        local = np.cumsum(dist.reshape(lanes, 64), axis=1, dtype=f32)[:, -1]
        incl = local.reshape(-1, 32).copy()
        for off in (1, 2, 4, 8, 16):
            step = incl.copy()
            step[:, off:] += incl[:, :-off]
            incl = step
        before = np.concatenate([[f32(0)], np.cumsum(incl[:, -1], dtype=f32)])
        total = before[-1]
        excl = (before[:-1, None] + np.concatenate([np.zeros((len(incl), 1), f32), incl[:, :-1]], axis=1)).reshape(-1)
        incl = (before[:-1, None] + incl).reshape(-1)
        target = f32(f32(unit(e + 1)) * total)
        at = n - 1
        if not total > 0:
            at = int(unit(e + 1) * n) % n
        hit = np.flatnonzero((excl <= target) & (target < incl))
        if total > 0 and len(hit):
            acc, run = excl[hit[0]], int(hit[0]) * 64
            at = run
            for k in range(run, min(run + 64, n)):
                if acc <= target:
                    at = k
                acc = f32(acc + dist[k])


@pytest.mark.parametrize("ic,bits", [(2, 6), (126, 6), (1024, 8), (1026, 6), (4096, 8), (4098, 6), (8190, 8), (8192, 8), (8194, 6)])
@pytest.mark.parametrize("kind", ["uniform", "ties"])
def test_mu_seeds_are_the_draws_of_the_definition(ic, bits, kind):
    """Vectors whose seeds are found from sums in a tree, with the chains behind them, up to 4096 of them (around the ends of runs, warps and of that
    range), against the chains; ties and zeros among the distances included."""
    rng = np.random.default_rng(ic + bits)
    mu16 = rng.uniform(0.0, 1.0, ic).astype(np.float16) if kind == "uniform" else (rng.integers(0, 9, ic) / 8.0).astype(np.float16)
    _, img = quantize_dev(mu16, B.RWKVQ_VQ, bits, seed=7, iters=0)
    _, codes = B.rwkvq_image_unpack(img.cpu().numpy())
    got = np.asarray(codes["codebook"]).reshape(1 << bits, 2).view(np.uint16)
    assert np.array_equal(got, _drawn_seeds(mu16.reshape(-1, 2), 1 << bits, 7).view(np.uint16))


@pytest.mark.parametrize("seed", [661793, 867062, 1253589])
def test_mu_seeds_where_one_vector_is_far_from_all_others(seed):
    """A thread's own sum of distances is thousands of times the target of the draw, which falls next to the boundary between two vectors."""
    i = np.arange(2048)
    v = np.stack([0.25 + (37 * i % 32) / 4096, 0.25 + (53 * i % 29) / 4096], axis=1)
    v[31] = 1.0
    v16 = v.astype(np.float16)
    _, img = quantize_dev(v16.reshape(-1), B.RWKVQ_VQ, 6, seed=seed, iters=0)
    _, codes = B.rwkvq_image_unpack(img.cpu().numpy())
    got = np.asarray(codes["codebook"]).reshape(64, 2).view(np.uint16)
    assert np.array_equal(got, _drawn_seeds(v16, 64, seed).view(np.uint16))


def test_quantize_dev_error_paths():
    w = torch.zeros((256, 256), dtype=torch.float16, device="cuda")
    ws = torch.empty(256, dtype=torch.uint8, device="cuda")
    d0 = B.rwkvq_desc_for(256, 256, B.RWKVQ_SQ, 3)
    img = torch.empty(int(d0.image_bytes) + 256, dtype=torch.uint8, device="cuda")
    with pytest.raises(B.RwkvqError) as e:
        B.rwkvq_quantize_dev(w, 256, 256, B.RWKVQ_SQ, 3, img[:1024], ws)
    assert e.value.status == 5
    with pytest.raises(B.RwkvqError) as e:
        B.rwkvq_quantize_dev(w, 256, 256, B.RWKVQ_SQ, 3, img[16:], ws)
    assert e.value.status == 3
    with pytest.raises(B.RwkvqError) as e:
        B.rwkvq_quantize_dev(w, 250, 256, B.RWKVQ_SQ, 3, img, ws)
    assert e.value.status == 2
    with pytest.raises(B.RwkvqError) as e:
        B.rwkvq_quantize_dev(w, 256, 256, B.RWKVQ_VQ, 6, img, ws, elem_weight=torch.ones(256, device="cuda"))
    assert e.value.status == 1
    for method, bits in ((B.RWKVQ_SQ, 3), (B.RWKVQ_VQ, 6)):
        bad = torch.zeros((256, 256), dtype=torch.float16, device="cuda")
        bad[200, 131] = float("nan")
        with pytest.raises(B.RwkvqError) as e:
            B.rwkvq_quantize_dev(bad, 256, 256, method, bits, img, ws)
        assert e.value.status == 4
    with pytest.raises(B.RwkvqError) as e:
        B.rwkvq_calib_representative(torch.zeros((1, 8), device="cuda"), 1.0, torch.zeros(8, device="cuda"))
    assert e.value.status == 1


@pytest.mark.parametrize("method,bits,oc,ic", [(B.RWKVQ_SQ, 3, 272, 384), (B.RWKVQ_SQ, 3, 512, 512), (B.RWKVQ_VQ, 6, 256, 512),
                                               (B.RWKVQ_VQ, 8, 256, 256)])
def test_quant_error_matches_oracle(method, bits, oc, ic):
    rng = np.random.default_rng(oc + ic + bits)
    w16 = (rng.standard_t(3, (oc, ic)) * 0.01).astype(np.float16)
    d, img = quantize_dev(w16, method, bits, seed=2, iters=3)
    _, codes = B.rwkvq_image_unpack(img.cpu().numpy())
    if method == B.RWKVQ_SQ:
        w_hat = orc.sq_decode(np.asarray(codes["q"]).reshape(oc, ic), np.asarray(codes["scale"]), np.asarray(codes["zero"]))
    else:
        w_hat = orc.vq_decode(np.asarray(codes["codebook"]).reshape(oc // 256, ic // 256, 1 << bits, 2),
                              np.asarray(codes["q"]).reshape(oc, ic // 2))
    wd = torch.from_numpy(w16).cuda()
    sse = B.rwkvq_quant_error(wd, d, img)
    ref = orc.quant_sse(w16, w_hat)
    assert abs(sse - ref) <= 1e-12 * ref
    assert sse == B.rwkvq_quant_error(wd, d, img)          # reproducible


def test_mse_selector_picks_the_smaller_error():
    # Section 5.3's "MSE" selector: code the matrix both ways, keep the coding with the smaller error
    rng = np.random.default_rng(77)
    for kind in ("gauss", "student"):
        w16 = ((rng.standard_normal((256, 512)) * 0.02) if kind == "gauss" else rng.standard_t(3, (256, 512)) * 0.01).astype(np.float16)
        wd = torch.from_numpy(w16).cuda()
        dq, iq = quantize_dev(w16, B.RWKVQ_SQ, 3)
        dv, iv = quantize_dev(w16, B.RWKVQ_VQ, 6, seed=1)
        e_sq, e_vq = B.rwkvq_quant_error(wd, dq, iq), B.rwkvq_quant_error(wd, dv, iv)
        q, s, z = orc.sq_encode(w16)
        assert abs(e_sq - orc.quant_sse(w16, orc.sq_decode(q, s, z))) <= 1e-12 * e_sq
        assert e_sq > 0.0 and e_vq > 0.0 and (e_sq < e_vq) == (orc.quant_sse(w16, orc.sq_decode(q, s, z)) < e_vq)


def test_async_quantizer_and_check():
    rng = np.random.default_rng(9)
    ws = torch.zeros(B.rwkvq_quantize_workspace_bytes(), dtype=torch.uint8, device="cuda")
    mats = [(rng.standard_normal((256, 384)) * 0.02).astype(np.float16) for _ in range(3)]
    imgs = []
    for w16 in mats:
        d0 = B.rwkvq_desc_for(256, 384, B.RWKVQ_SQ, 3)
        img = torch.empty(int(d0.image_bytes), dtype=torch.uint8, device="cuda")
        B.rwkvq_quantize_dev_async(torch.from_numpy(w16).cuda(), 256, 384, B.RWKVQ_SQ, 3, img, ws)
        imgs.append(img)
    assert B.rwkvq_quantize_check(ws) == 0
    for w16, img in zip(mats, imgs):
        ref = B.rwkvq_pack(w16, 256, 384, B.RWKVQ_SQ, 3).image()
        assert np.array_equal(img.cpu().numpy()[256:], ref[256:])
    bad = mats[1].copy()
    bad[7, 300] = np.float16(np.inf)
    for w16 in (mats[0], bad, mats[2]):           # the flag of the middle call survives the later one
        B.rwkvq_quantize_dev_async(torch.from_numpy(w16).cuda(), 256, 384, B.RWKVQ_SQ, 3, imgs[0], ws)
    assert B.rwkvq_quantize_check(ws) == 4
    assert B.rwkvq_quantize_check(ws) == 0        # cleared by the check


def _edge_tile(kind):
    rng = np.random.default_rng(77)
    if kind == "constant":
        return np.full((256, 256), -0.125, np.float16)
    if kind == "few":
        return rng.choice(np.array([-1.5, -0.0, 0.0, 2.0 ** -24, 0.75, 60000.0], np.float16), (256, 256))
    if kind == "wide":              # magnitudes over the whole range, a few vectors far out on each side
        return (rng.choice([-1.0, 1.0], (256, 256)) * np.exp(rng.uniform(np.log(1e-7), np.log(6e4), (256, 256)))).astype(np.float16)
    if kind == "offset":            # all of one sign, far from zero
        return (rng.standard_normal((256, 256)) * 0.01 + 3.0).astype(np.float16)
    return (rng.standard_t(3, (256, 256)) * 0.01).astype(np.float16)


@pytest.mark.parametrize("bits", [6, 8])
@pytest.mark.parametrize("kind", ["constant", "few", "wide", "offset", "tails"])
def test_vq_device_iterations_and_assignment_at_the_edges(kind, bits):
    """Candidate lists and cluster sums: the assignment is the nearest centre of all, and one iteration moves the seeds to the
    means of their members."""
    w16 = _edge_tile(kind)
    v = tile_vectors(w16, 0, 0)
    books = []
    for iters in (0, 1, 7):
        _, img = quantize_dev(w16, B.RWKVQ_VQ, bits, seed=9, iters=iters)
        _, codes = B.rwkvq_image_unpack(img.cpu().numpy())
        c = np.asarray(codes["codebook"]).reshape(1 << bits, 2).astype(np.float64)
        assert np.array_equal(np.asarray(codes["q"]).reshape(-1), orc._nearest(v, c)), (kind, iters)
        books.append(c)
    near = orc._nearest(v, books[0])
    for e in range(1 << bits):
        members = v[near == e]
        want = members.mean(axis=0) if len(members) else books[0][e]
        # fp16 rounding; a tie decided otherwise in fp32 moves a mean by less than that of a cluster's spread
        assert np.all(np.abs(books[1][e] - want) <= 1e-3 * np.abs(want) + 2.0 ** -24 + 1e-2 * (np.ptp(members, axis=0) if len(members) else 0.0)), (kind, e)


@pytest.mark.parametrize("bits", [6, 8])
@pytest.mark.parametrize("few", [1, 33, 34, 66, 67, 100])
def test_vq_tiles_alike_in_one_block_and_in_a_cluster(few, bits):
    """101 tiles are taken by a block each, up to 100 by clusters of four (at 33 and 66 with other blocks on an SM): the first tiles of a wide
    matrix come out alike, with weights beyond the two-piece sums and many equal ones among them, and as the oracle assigns them."""
    rng = np.random.default_rng(few)
    w16 = (rng.standard_t(3, (256, 101 * 256)) * 0.01).astype(np.float16)
    w16[:, 256:512] *= np.float16(900.0)              # around four in magnitude, on both sides
    w16[:, 512:768] = rng.choice(np.array([-0.5, 0.0, 2.0 ** -24, 3.0], np.float16), (256, 256))
    _, wide = quantize_dev(w16, B.RWKVQ_VQ, bits, seed=11, iters=4)
    _, part = quantize_dev(w16[:, :few * 256], B.RWKVQ_VQ, bits, seed=11, iters=4)
    E = 1 << bits
    books, index = [], []
    for img, tiles in ((wide, 101), (part, few)):
        _, codes = B.rwkvq_image_unpack(img.cpu().numpy())
        books.append(np.asarray(codes["codebook"]).reshape(tiles, E, 2)[:few])
        index.append(np.asarray(codes["q"]).reshape(256, tiles * 128)[:, :few * 128])
    assert np.array_equal(books[0].view(np.uint16), books[1].view(np.uint16))
    assert np.array_equal(index[0], index[1])
    for t in range(min(few, 3)):
        v = w16[:, t * 256:(t + 1) * 256].astype(np.float64).reshape(-1, 2)
        assert np.array_equal(index[1][:, t * 128:(t + 1) * 128].reshape(-1), orc._nearest(v, books[1][t].astype(np.float64)))


@pytest.mark.parametrize("oc,ic,bits", [(128, 256, 3), (2048, 1024, 3), (256, 512, 6), (2816, 2816, 6), (1, 1024, 6), (1, 10240, 8)])
def test_quantizers_start_behind_what_writes_their_inputs(oc, ic, bits):
    """Kernels that write the weights, quantize them, read the image and write other weights, one behind the other without a wait of the host."""
    method = B.RWKVQ_SQ if bits == 3 else B.RWKVQ_VQ
    desc = B.rwkvq_desc_for(oc, ic, method, bits)
    ws = torch.zeros(B.rwkvq_quantize_workspace_bytes(), dtype=torch.uint8, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(oc + ic)
    src = [(torch.randn((oc, ic), generator=g, device="cuda") * 0.02).half() for _ in range(4)]
    samples = [torch.randn((40, ic), generator=g, device="cuda") for _ in range(4)]
    w, image = torch.zeros((oc, ic), dtype=torch.float16, device="cuda"), torch.zeros(int(desc.image_bytes), dtype=torch.uint8, device="cuda")
    rep, out = torch.zeros(ic, device="cuda"), torch.empty((oc, ic), device="cuda")

    def one(i, wait):
        for step in (lambda: w.copy_(src[i]), lambda: B.rwkvq_calib_representative(samples[i], 1.0, rep_sq=rep),
                     lambda: B.rwkvq_quantize_dev_async(w, oc, ic, method, bits, image, ws, elem_weight=rep if oc == 1 else None, kmeans_iters=2, seed=i),
                     lambda: B.rwkvq_dequant(desc, image, out)):
            step()
            if wait:
                torch.cuda.synchronize()
        return out.clone()

    want = [one(i, True) for i in range(4)]
    got = [one(i % 4, False) for i in range(16)]
    assert B.rwkvq_quantize_check(ws) == 0
    for i, y in enumerate(got):
        assert torch.equal(y, want[i % 4])


@pytest.mark.parametrize("reader,oc", [("samples", 2048), ("scalar", 1024), ("tile", 512), ("tile", 26112), ("vector", 1024), ("vector", 10240)])
def test_quantizers_behind_products_that_end_late(reader, oc):
    """What a product writes is quantized at once.  The products' kernels let the next one start when they do, so the quantizer is resident while they
    write; every call changes all of the buffer."""
    ic, rows = 512, 1 if reader == "vector" else 256
    ws = torch.zeros(B.rwkvq_quantize_workspace_bytes(), dtype=torch.uint8, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(oc)
    desc = B.rwkvq_desc_for(oc, ic, B.RWKVQ_SQ, 3)
    W = torch.zeros(int(desc.image_bytes), dtype=torch.uint8, device="cuda")
    B.rwkvq_quantize_dev_async((torch.randn((oc, ic), generator=g, device="cuda") * 0.02).half(), oc, ic, B.RWKVQ_SQ, 3, W, ws)
    x = [torch.randn((rows, ic), generator=g, device="cuda").to(torch.float16 if rows == 1 else torch.bfloat16) for _ in range(4)]
    y = torch.zeros((rows, oc), device="cuda", dtype=torch.float16 if rows == 1 else torch.float32 if reader == "samples" else torch.bfloat16)
    pws = torch.zeros(max(256, B.rwkvq_gemv_workspace_bytes(desc, 1), B.rwkvq_prefill_workspace_bytes(desc, rows, False)), dtype=torch.uint8, device="cuda")
    method, bits = (B.RWKVQ_SQ, 3) if reader == "scalar" else (B.RWKVQ_VQ, 6)
    image_desc = None if reader == "samples" else B.rwkvq_desc_for(rows, oc, method, bits)
    image = torch.zeros(oc * 4 if image_desc is None else int(image_desc.image_bytes), dtype=torch.uint8, device="cuda")

    def one(i, wait):
        if rows == 1:
            B.rwkvq_gemv(desc, W, None, None, x[i], None, 1, y, pws)
        else:
            B.rwkvq_gemm_prefill(desc, W, None, None, x[i], None, rows, y, pws)
        if wait:
            torch.cuda.synchronize()
        if reader == "samples":
            B.rwkvq_calib_representative(y, 1.0, rep=image.view(torch.float32))
        else:       # the bit patterns of bf16 results of this size are finite fp16 numbers
            B.rwkvq_quantize_dev_async(y.view(torch.float16), rows, oc, method, bits, image, ws, kmeans_iters=1, seed=i)
        return image.clone()

    want = [one(i, True) for i in range(4)]
    got = [one(i % 4, False) for i in range(24)]
    assert B.rwkvq_quantize_check(ws) == 0
    assert not torch.equal(want[0], want[1])
    for i, z in enumerate(got):
        assert torch.equal(z, want[i % 4])


@pytest.mark.parametrize("oc,ic,bits", [(512, 512, 3), (4096, 4096, 3), (512, 512, 6), (512, 512, 8), (2816, 2816, 6), (1, 512, 6), (1, 10240, 8)])
def test_products_behind_quantizers(oc, ic, bits):
    """A product reads the image that the quantizer in front of it is still writing when it starts: one image buffer, other weights every time."""
    method = B.RWKVQ_SQ if bits == 3 else B.RWKVQ_VQ
    desc = B.rwkvq_desc_for(oc, ic, method, bits)
    ws = torch.zeros(B.rwkvq_quantize_workspace_bytes(), dtype=torch.uint8, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(oc + 3 * ic)
    src = [(torch.rand((oc, ic), generator=g, device="cuda") - 0.5).half() for _ in range(4)]
    image = torch.zeros(int(desc.image_bytes), dtype=torch.uint8, device="cuda")
    pdesc, pimage, rows = desc, image, oc
    if oc == 1:      # a token-shift vector: the product's matrix stays as it is
        rows = 512
        pdesc = B.rwkvq_desc_for(rows, ic, B.RWKVQ_SQ, 3)
        pimage = torch.zeros(int(pdesc.image_bytes), dtype=torch.uint8, device="cuda")
        B.rwkvq_quantize_dev_async((torch.randn((rows, ic), generator=g, device="cuda") * 0.02).half(), rows, ic, B.RWKVQ_SQ, 3, pimage, ws)
    x, xprev = torch.randn((3, ic), generator=g, device="cuda").half(), torch.randn((3, ic), generator=g, device="cuda").half()
    y, pws = torch.zeros((3, rows), device="cuda"), torch.zeros(max(256, B.rwkvq_gemv_workspace_bytes(pdesc, 3)), dtype=torch.uint8, device="cuda")

    def one(i, wait):
        B.rwkvq_quantize_dev_async(src[i], oc, ic, method, bits, image, ws, kmeans_iters=1, seed=i)
        if wait:
            torch.cuda.synchronize()
        mu = (desc, image, x, xprev) if oc == 1 else (None, None, x, None)
        B.rwkvq_gemv(pdesc, pimage, *mu, 3, y, pws)
        return y.clone()

    want = [one(i, True) for i in range(4)]
    got = [one(i % 4, False) for i in range(24)]
    assert B.rwkvq_quantize_check(ws) == 0
    assert not torch.equal(want[0], want[1])
    for i, z in enumerate(got):
        assert torch.equal(z, want[i % 4])


@pytest.mark.parametrize("oc,ic,bits", [(256, 512, 3), (512, 512, 6), (2816, 2816, 8), (1, 1024, 6), (1, 10240, 6)])
def test_captured_quantizers(oc, ic, bits):
    """A graph of the weights' copy, the representative and the quantizer gives the images of the calls made one by one."""
    method = B.RWKVQ_SQ if bits == 3 else B.RWKVQ_VQ
    desc = B.rwkvq_desc_for(oc, ic, method, bits)
    ws = torch.zeros(B.rwkvq_quantize_workspace_bytes(), dtype=torch.uint8, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(oc * 7 + ic)
    src = [(torch.randn((oc, ic), generator=g, device="cuda") * 0.02).half() for _ in range(3)]
    samples = torch.randn((33, ic), generator=g, device="cuda")
    fresh, w, rep = torch.zeros_like(src[0]), torch.zeros_like(src[0]), torch.zeros(ic, device="cuda")
    image = torch.zeros(int(desc.image_bytes), dtype=torch.uint8, device="cuda")

    def calls():
        w.copy_(fresh)
        B.rwkvq_calib_representative(samples, 1.0, rep_sq=rep)
        B.rwkvq_quantize_dev_async(w, oc, ic, method, bits, image, ws, elem_weight=rep if oc == 1 else None, kmeans_iters=2, seed=5)

    want = []
    for s in src:
        fresh.copy_(s)
        calls()
        want.append(image.clone())
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls()
    for s, ref in list(zip(src, want)) * 2:
        fresh.copy_(s)
        image.zero_()
        graph.replay()
        assert torch.equal(image, ref)
    assert B.rwkvq_quantize_check(ws) == 0


@pytest.mark.parametrize("oc,ic,bits,weighted", [(256, 256, 6, False), (512, 768, 8, False), (1, 128, 6, False), (1, 4096, 6, True), (1, 10240, 8, False)])
@pytest.mark.parametrize("mute", [0, 1, 3])
def test_waits_between_blocks_run_out(oc, ic, bits, weighted, mute):
    """A block of every cluster sends nothing: the others give up, the kernels return, the next check reports ETIMEOUT once, and the calls after it are right."""
    g = torch.Generator(device="cuda").manual_seed(ic + bits)
    w = (torch.randn((oc, ic), generator=g, device="cuda") * 0.02).half()
    weight = torch.rand(ic, generator=g, device="cuda") if weighted else None
    desc = B.rwkvq_desc_for(oc, ic, B.RWKVQ_VQ, bits)
    ws = torch.zeros(B.rwkvq_quantize_workspace_bytes(), dtype=torch.uint8, device="cuda")
    image, again = (torch.zeros(int(desc.image_bytes), dtype=torch.uint8, device="cuda") for _ in range(2))
    B.rwkvq_quantize_dev_async(w, oc, ic, B.RWKVQ_VQ, bits, image, ws, elem_weight=weight, kmeans_iters=3, seed=2)
    assert B.rwkvq_quantize_check(ws) == 0
    B.rwkvq_quantize_dev_lost(w, oc, ic, B.RWKVQ_VQ, bits, again, ws, 200, mute, elem_weight=weight, kmeans_iters=3, seed=2)
    B.rwkvq_quantize_dev_async(w, oc, ic, B.RWKVQ_VQ, bits, again, ws, elem_weight=weight, kmeans_iters=3, seed=2)
    assert B.rwkvq_quantize_check(ws) == 8 and B.rwkvq_quantize_check(ws) == 0
    assert torch.equal(image, again)
