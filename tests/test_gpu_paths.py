"""Kernels that are chosen by shape or alignment against the general path or plain
arithmetic: the block-aligned search against the general search kernels (bit-equal),
power-of-two downsampling, the stage-2 ring of the sub-band sums, the split of a wide
band between the byte and the tensor-core kernel, and a training step's layers."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gsp():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2110_12749_gb300 import build, gsp as g
    build.build()
    g.lib()
    return g


def _series(rows, n, seed):
    """Noise with drifts, a constant block, a loud block, pulses across block ends and a
    row of zeros."""
    rng = np.random.default_rng(seed)
    t = np.arange(n)
    D = rng.normal(40000.0, 300.0, (rows, n)) + 200.0 * np.sin(t / 300.0)
    for r in range(rows):
        for b in range(1024, n, 1024):
            w = int(rng.integers(1, 150))
            t0 = b - int(rng.integers(0, w + 1))
            D[r, t0:t0 + w] += 9.0 * 300.0 / np.sqrt(w)
    if n >= 4096:
        D[0, 1024:2048] = 40000
        D[1 % rows, 2048:3072] += rng.normal(0, 3000.0, 1024)
    D[-1] = 0
    return np.rint(D).astype(np.int32)


@pytest.mark.parametrize("rows,n,t_offset,threshold", [
    (1, 1024, 0, 2.0), (3, 2047, 0, 2.0), (5, 4096, 1024, 3.0), (7, 17 * 1024 + 5, -3072, 4.0),
    (2, 40 * 1024, 5 * 1024, -1.0), (4, 6000, 0, 1e9)])
def test_block_aligned_search_equals_general(gsp, rows, n, t_offset, threshold):
    D = _series(rows, n, rows)
    d, keep = gsp.make_desc(32, 1200.0, 1500.0, 1e-4, n, ndm=rows, dm_step=0.0, threshold=threshold)
    plan = gsp.gsp_plan_create(d, keep)
    got = []
    for shift in (0, 1):   # a row start off the 16-byte boundary takes the general kernels
        buf = torch.zeros(rows * ((n + 7) // 4 * 4) + 4, dtype=torch.int32, device="cuda")
        v = buf[shift:shift + rows * ((n + 7) // 4 * 4)].view(rows, -1)
        v[:, :n] = torch.from_numpy(D).cuda()
        gsp.gsp_search_series(plan, v, n, t_offset)
        c, total, _ = gsp.gsp_candidates(plan)
        st = gsp.gsp_search_stats(plan, n)
        got.append((c.copy(), total, st))
    (a, na, sa), (b, nb, sb) = got
    assert na == nb and (a == b).all()
    assert (sa["sigma_b"] == sb["sigma_b"]).all() and (sa["bad"] == sb["bad"]).all()


@pytest.mark.parametrize("ds", [2, 4, 8, 16, 32, 64, 128])
@pytest.mark.parametrize("n_in,pad", [(16, 0), (1000, 8), (4096, 0), (16384 + 77, 3)])
def test_downsample_powers_of_two(gsp, ds, n_in, pad):
    rng = np.random.default_rng(ds)
    C, n = 3, n_in // ds
    x = rng.integers(0, 256, (C, (n_in + 15) // 16 * 16), dtype=np.uint8)
    x[0, :] = 255
    out = torch.full((C, (n + 7) // 8 * 8 + 8 + pad), 7, dtype=torch.uint8, device="cuda")
    gsp.gsp_downsample(torch.from_numpy(x).cuda(), C, n_in, ds, out)
    s = x[:, :n * ds].reshape(C, n, ds).astype(np.int64).sum(2)
    ref = (2 * s + ds) // (2 * ds)
    o = out.cpu().numpy()
    assert (o[:, :n] == ref).all() and (o[:, n:] == 7).all()


@pytest.mark.parametrize("nchan,nsub,group,ndm,step,n_in", [
    (60, 5, 3, 10, 2.0, 3000), (64, 64, 16, 33, 1.0, 4000), (96, 1, 12, 25, 0.5, 2600), (48, 6, 1, 4, 20.0, 5000)])
def test_subband_sums(gsp, nchan, nsub, group, ndm, step, n_in):
    d, keep = gsp.make_desc(nchan, 1200.0, 1500.0, 1e-4, n_in, ndm=ndm, dm_lo=3.0, dm_step=step)
    sub = gsp.gsp_subband_create(d, nsub, group)
    d1, d2, _ = gsp.gsp_subband_delays(sub)
    n = gsp.gsp_subband_nout(sub, n_in)
    x = np.random.default_rng(nsub).integers(0, 256, (nchan, (n_in + 15) // 16 * 16), dtype=np.uint8)
    out = torch.full((ndm, (n + 3) // 4 * 4 + 4), -7, dtype=torch.int32, device="cuda")
    gsp.gsp_subband_dedisperse(sub, torch.from_numpy(x).cuda(), n_in, out)
    gsp.gsp_subband_finish(sub)
    ref = np.zeros((ndm, n), np.int64)
    cs = nchan // nsub
    for k in range(ndm):
        for c in range(nchan):
            o = d1[k // group, c] + d2[k, c // cs]
            ref[k] += x[c, o:o + n]
    o = out.cpu().numpy()
    assert (o[:, :n] == ref).all() and (o[:, n:] == -7).all()


@pytest.mark.parametrize("descending", [False, True])
def test_wide_band_split_bit_exact(gsp, orc, monkeypatch, descending):
    monkeypatch.delenv("GSP_DD_VARIANT", raising=False)
    nchan, ndm, n_out = 1024, 240, 50001
    dl, _ = orc.delays(nchan, 500.0, 3300.0, 98.304e-6, np.arange(ndm) * 1.0)
    if descending:
        dl = np.ascontiguousarray(dl[:, ::-1])
    n_in = n_out + orc.max_delay(dl)
    x = np.random.default_rng(5).integers(0, 256, (nchan, (n_in + 15) // 16 * 16), dtype=np.uint8)
    d, keep = gsp.make_desc(nchan, 500.0, 3300.0, 98.304e-6, n_in, ndm=ndm, dm_step=1.0,
                            freq_descending=descending)
    plan = gsp.gsp_plan_create(d, keep)
    xd = torch.from_numpy(x).cuda()
    out = torch.full((ndm, (n_out + 3) // 4 * 4), -7, dtype=torch.int32, device="cuda")
    gsp.gsp_dedisperse(plan, xd, n_in, out)
    assert gsp.gsp_plan_launches(plan) == 2      # byte kernel and tensor-core kernel
    assert (out.cpu().numpy()[:, :n_out] == orc.dedisperse(x, n_in, dl)).all()
    gsp.gsp_search(plan, xd, n_in)
    s1 = gsp.gsp_search_stats(plan, n_out)
    gsp.gsp_search_series(plan, out, n_out)
    s2 = gsp.gsp_search_stats(plan, n_out)
    assert (s1["sigma_b"] == s2["sigma_b"]).all()


@pytest.mark.parametrize("n", [1, 5, 33])
def test_training_layers_consistent(gsp, n):
    """Pool, its way back and the weight and bias gradients of each conv layer from the
    tensors that the step keeps, in 64 bits."""
    rng = np.random.default_rng(n)
    r = gsp.gsp_ranker_create(n, 3)
    x = torch.from_numpy(rng.normal(0, 1, (n, 64, 64)).astype(np.float32)).cuda()
    y = torch.from_numpy(rng.integers(0, 2, n).astype(np.int32)).cuda()
    gsp.gsp_ranker_train_step(r, x, y, n, 0.0)
    gsp.gsp_ranker_finish(r)
    _, g = gsp.gsp_ranker_get_params(r)
    bf = lambda v: torch.from_numpy(np.asarray(v, np.float32)).bfloat16().double().numpy()  # noqa: E731
    act, at = bf(x.cpu().numpy())[..., None], 0
    for l, (cin, cout, side) in enumerate([(1, 8, 64), (8, 16, 32), (16, 32, 16)]):
        h = side // 2
        t = {k: gsp.gsp_ranker_tensor(r, k + str(l)) for k in ("z", "a", "idx", "ga", "gz")}
        z = t["z"].reshape(n, h, 2, h, 2, cout).transpose(0, 1, 3, 5, 2, 4).reshape(n, h, h, cout, 4)
        assert (t["idx"].reshape(n, h, h, cout) == z.argmax(-1)).all()
        assert (t["a"].reshape(n, h, h, cout) == bf(z.max(-1))).all()
        v = np.where(z.max(-1) > 0, t["ga"].reshape(n, h, h, cout), 0.0)
        gz = np.zeros((n, h, h, cout, 4))
        np.put_along_axis(gz, z.argmax(-1)[..., None], bf(v)[..., None], -1)
        gz = gz.reshape(n, h, h, cout, 2, 2).transpose(0, 1, 4, 2, 5, 3).reshape(n, side, side, cout)
        assert (t["gz"].reshape(n, side, side, cout) == gz).all()
        p = np.pad(act, ((0, 0), (1, 1), (1, 1), (0, 0)))
        dw, mag = np.zeros((cout, cin, 3, 3)), np.zeros((cout, cin, 3, 3))
        for ky in range(3):
            for kx in range(3):
                s = p[:, ky:ky + side, kx:kx + side]
                dw[:, :, ky, kx] = np.einsum("bijo,bijc->oc", gz, s)
                mag[:, :, ky, kx] = np.einsum("bijo,bijc->oc", abs(gz), abs(s))
        k = n * side * side // 4      # nonzero terms of a sum: one per pooling window
        got = g[at:at + dw.size].reshape(dw.shape)
        assert (abs(got - dw) <= (k + 8) * 2.0 ** -24 * mag + 1e-30).all()
        at += dw.size
        db = v.sum((0, 1, 2))
        assert (abs(g[at:at + cout] - db) <= (k + 8) * 2.0 ** -24 * abs(v).sum((0, 1, 2)) + 1e-30).all()
        at += cout
        act = t["a"].reshape(n, h, h, cout)


@pytest.mark.parametrize("n,c,pad,off,out_off", [
    (256, 320, 0, 0, 0),     # five channel tiles: a group of four and one alone
    (257, 321, 2, 1, 0),     # input words shifted by 1, 2 and 3 bytes
    (255, 80, 3, 2, 0),
    (1, 16, 0, 3, 0),        # the only words would reach outside the matrix
    (2, 17, 0, 0, 0),
    (1030, 706, 0, 0, 0),
    (513, 130, 4, 0, 0),
    (300, 260, 16, 0, 1),    # output not aligned: the kernel of byte and word accesses
])
def test_ingest_alignments(gsp, n, c, pad, off, out_off):
    rng = np.random.default_rng(n * c + off)
    flat = torch.from_numpy(rng.integers(0, 256, n * (c + pad) + off, dtype=np.uint8)).cuda()
    x = flat[off:].view(n, c + pad)
    stride = (n + 15) // 16 * 16 + 16
    buf = torch.full((c * stride + out_off,), 7, dtype=torch.uint8, device="cuda")
    out = buf[out_off:].view(c, stride)
    gsp.gsp_ingest_transpose(x, n, c, out)
    assert torch.equal(out[:, :n], x[:, :c].t())
    assert bool((out[:, n:] == 7).all()) and bool((buf[:out_off] == 7).all())
