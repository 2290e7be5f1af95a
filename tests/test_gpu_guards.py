"""Calls at the edges of what the kernels' guards cover: orders of barriers and waits
under repetition, positions and sums near the ends of their number ranges, kernels that are
chosen for a call although the plan has another, waits that run out, and plans and objects
that are used side by side."""
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


def _status(gsp, call):
    try:
        call()
    except gsp.GspError as e:
        return e.status
    return gsp.GSP_OK


@pytest.mark.parametrize("rows,nblk", [(600, 40), (5000, 2), (300, 33)])
def test_block_aligned_search_repeats(gsp, rows, nblk):
    """Several blocks per CTA and a candidate in every window: each pass of the
    block-aligned search equals the general kernels' (rows off the 16-byte boundary)."""
    n = nblk * 1024
    g = torch.Generator(device="cuda")
    g.manual_seed(rows)
    D = torch.empty((rows, n), device="cuda").normal_(50000.0, 400.0, generator=g).round_().to(torch.int32)
    d, keep = gsp.make_desc(32, 1200.0, 1500.0, 1e-4, n, ndm=rows, dm_step=0.0, threshold=0.0)
    plan = gsp.gsp_plan_create(d, keep)
    flat = torch.zeros(rows * n + 4, dtype=torch.int32, device="cuda")
    off = flat[1:1 + rows * n].view(rows, n)
    off.copy_(D)
    gsp.gsp_search_series(plan, off, n)
    want, total, _ = gsp.gsp_candidates(plan)
    assert total == rows * nblk
    for _ in range(8):
        gsp.gsp_search_series(plan, D, n)
        got, m, _ = gsp.gsp_candidates(plan)
        assert m == total and (got == want).all()


@pytest.mark.parametrize("nchan,ndm,n_in", [(512, 32, 1 << 20), (24, 40, 1 << 21), (100, 16, 1 << 21), (9, 33, 1 << 20)])
def test_tensor_core_dedispersion_repeats(gsp, monkeypatch, nchan, ndm, n_in):
    """Rings of a few chunks per item, inputs cold in L2 and far apart: every pass of the
    tensor-core kernel equals the byte kernel."""
    g = torch.Generator(device="cuda")
    g.manual_seed(nchan)
    x = torch.randint(0, 256, (nchan, n_in), dtype=torch.uint8, device="cuda", generator=g)
    cold = torch.empty(1 << 28, dtype=torch.uint8, device="cuda")
    want = None
    for variant in (32, gsp.gsp_dedisperse_variants()[0] - 1):
        monkeypatch.setenv("GSP_DD_VARIANT", str(variant))
        d, keep = gsp.make_desc(nchan, 1200.0, 1500.0, 1e-4, n_in, ndm=ndm, dm_step=0.7, block_len=4096)
        plan = gsp.gsp_plan_create(d, keep)
        assert gsp.gsp_dedisperse_variants(plan)[1] == variant
        n_out = gsp.gsp_plan_nout(plan, n_in)
        out = torch.zeros((ndm, (n_out + 3) // 4 * 4), dtype=torch.int32, device="cuda")
        for _ in range(1 if want is None else 25):
            out.zero_()
            cold.fill_(1)
            gsp.gsp_dedisperse(plan, x, n_in, out)
            if want is None:
                want = out.clone()
            assert torch.equal(out, want)


@pytest.mark.parametrize("first", [(1 << 30) - 600, (1 << 30) + 12345, (1 << 31) - 100])
def test_delays_beyond_30_bits(gsp, monkeypatch, first):
    """Delays around 2^30 samples and up to the largest one accepted, trials close together
    (so that the tensor-core kernel takes them): the sums of two channels, exactly."""
    monkeypatch.setenv("GSP_DD_VARIANT", str(gsp.gsp_dedisperse_variants()[0] - 1))
    ndm, n_out = 17, 5000
    delays = np.zeros((ndm, 2), np.int32)
    delays[:, 0] = first + 5 * np.arange(ndm)
    n_in = int(delays.max()) + n_out
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    x = torch.randint(0, 256, (2, (n_in + 15) // 16 * 16), dtype=torch.uint8, device="cuda", generator=g)
    d, keep = gsp.make_desc(2, 1200.0, 1500.0, 1e-4, n_in, delays=delays, block_len=1 << 16,
                            window_len=1 << 20, max_cands=16)
    plan = gsp.gsp_plan_create(d, keep)
    assert gsp.gsp_dedisperse_variants(plan)[1] == gsp.gsp_dedisperse_variants()[0] - 1
    out = torch.full((ndm, n_out), -7, dtype=torch.int32, device="cuda")
    gsp.gsp_dedisperse(plan, x, n_in, out)
    for i in range(ndm):
        a = int(delays[i, 0])
        assert torch.equal(out[i], x[0, a:a + n_out].int() + x[1, :n_out].int()), i


@pytest.mark.parametrize("nchan,values", [
    (65793, (255, 255)),     # the most channels the kernel takes: 2^24 - 1 in every sample
    (65792, (251, 255)),
    (50001, (128, 255)),     # sums above 2^23 whose low bits vary
    (33000, (254, 255)),
    (65793, (0, 1)),
])
@pytest.mark.parametrize("descending", [False, True])
def test_tensor_core_sums_to_24_bits(gsp, monkeypatch, nchan, values, descending):
    """The FP32 accumulators hold whole numbers below 2^24: sums up to the limit are exact,
    and so are the block sums taken from them."""
    mma = gsp.gsp_dedisperse_variants()[0] - 1
    monkeypatch.setenv("GSP_DD_VARIANT", str(mma))
    ndm, n_out = 17, 2100
    pos = np.arange(nchan) if descending else np.arange(nchan)[::-1]
    delays = (pos[None, :] * (3 + np.arange(ndm)[:, None]) // 16384).astype(np.int32)
    n_in = n_out + int(delays.max())
    g = torch.Generator(device="cuda")
    g.manual_seed(nchan)
    x = torch.randint(values[0], values[1] + 1, (nchan, (n_in + 15) // 16 * 16), dtype=torch.uint8,
                      device="cuda", generator=g)
    d, keep = gsp.make_desc(nchan, 1200.0, 1500.0, 1e-4, n_in, delays=delays, freq_descending=descending)
    plan = gsp.gsp_plan_create(d, keep)
    assert gsp.gsp_dedisperse_variants(plan)[1] == mma
    out = torch.full((ndm, n_out), -7, dtype=torch.int32, device="cuda")
    gsp.gsp_search(plan, x, n_in, 0, out)
    fused = gsp.gsp_search_stats(plan, n_out)
    for i in range(ndm):
        ref = torch.zeros(n_out, dtype=torch.int64, device="cuda")
        for v in np.unique(delays[i]):
            c = np.nonzero(delays[i] == v)[0]
            ref += x[c[0]:c[-1] + 1, int(v):int(v) + n_out].sum(0, dtype=torch.int64)
        assert torch.equal(out[i].long(), ref), i
    gsp.gsp_search_series(plan, out, n_out)
    plain = gsp.gsp_search_stats(plan, n_out)
    assert (fused["sigma_b"] == plain["sigma_b"]).all() and (fused["bad"] == plain["bad"]).all()


def test_autotuned_batch_with_short_blocks(gsp, monkeypatch):
    """Plans on a byte variant whose batch is tuned to the tensor-core kernel, with search blocks
    that the byte variant sums on the way and the tensor-core kernel does not."""
    nchan, block, mma = 1024, 800, gsp.gsp_dedisperse_variants()[0] - 1
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    plans, refs, xs, n_ins = [], [], [], []
    for n_in, ndm in [(100000, 256), (90000, 240)]:
        def make():
            d, keep = gsp.make_desc(nchan, 1000.0, 1500.0, 49.152e-6, n_in, ndm=ndm, dm_step=0.25,
                                    block_len=block, threshold=4.0)
            return gsp.gsp_plan_create(d, keep)
        monkeypatch.setenv("GSP_DD_VARIANT", "32")
        plans.append(make())
        assert gsp.gsp_dedisperse_variants(plans[-1])[1] == 32
        monkeypatch.delenv("GSP_DD_VARIANT")
        refs.append(make())
        xs.append(torch.randint(0, 256, (nchan, (n_in + 15) // 16 * 16), dtype=torch.uint8,
                                device="cuda", generator=g))
        n_ins.append(n_in)
    b = gsp.gsp_batch_create(plans, gsp.GSP_BATCH_PERSISTENT | gsp.GSP_BATCH_AUTOTUNE)
    for _ in range(2):
        gsp.gsp_batch_search(b, xs, n_ins)
        got, n, st = gsp.gsp_batch_candidates(b)
        assert st == gsp.GSP_OK and n > 0
    assert mma in [v for v, _ in gsp.gsp_batch_tune_results(b)]
    assert gsp.gsp_batch_info(b)[0] == mma   # 1.5 times faster than any byte variant here
    off = 0
    for i, (p, ref, x, n_in) in enumerate(zip(plans, refs, xs, n_ins)):
        gsp.gsp_search(ref, x, n_in)
        want, m, _ = gsp.gsp_candidates(ref)
        mine = got[off:off + m]
        off += m
        assert (mine["beam"] == i).all()
        for f in ("dm_idx", "t", "width", "snr"):
            assert (mine[f] == want[f]).all(), (i, f)
        n_out = gsp.gsp_plan_nout(p, n_in)
        assert (gsp.gsp_search_stats(p, n_out)["sigma_b"] == gsp.gsp_search_stats(ref, n_out)["sigma_b"]).all()
    assert off == n


@pytest.mark.parametrize("cycles,starve", [(2_000_000, 1), (3000, 0), (1, 0)])
def test_tensor_core_waits_that_run_out(gsp, monkeypatch, cycles, starve):
    """Nothing copied: a timeout.  Limits shorter than a frame of products, or than any copy (a
    wait always tests its barrier twice and may sleep in between, so it can still succeed): a
    timeout or exact sums.  The plan then gives exact sums."""
    monkeypatch.setenv("GSP_DD_VARIANT", str(gsp.gsp_dedisperse_variants()[0] - 1))
    nchan, n_in, ndm = 512, 100000, 40
    d, keep = gsp.make_desc(nchan, 1200.0, 1500.0, 1e-4, n_in, ndm=ndm, dm_step=1.0)
    plan = gsp.gsp_plan_create(d, keep)
    assert gsp.gsp_dedisperse_variants(plan)[1] == gsp.gsp_dedisperse_variants()[0] - 1
    g = torch.Generator(device="cuda")
    g.manual_seed(4)
    x = torch.randint(0, 256, (nchan, n_in), dtype=torch.uint8, device="cuda", generator=g)
    dl = gsp.gsp_plan_delays(plan)
    n_out = gsp.gsp_plan_nout(plan, n_in)
    out = torch.zeros((ndm, (n_out + 3) // 4 * 4), dtype=torch.int32, device="cuda")
    ref = {i: sum(x[c, int(dl[i, c]):int(dl[i, c]) + n_out].int() for c in range(nchan))
           for i in (0, 17, ndm - 1)}
    for limit in [(cycles, starve), (4_000_000_000, 0)] * 3:
        gsp.gsp_plan_set_wait_limit(plan, *limit)
        gsp.gsp_search(plan, x, n_in, 0, out)
        status = _status(gsp, lambda: gsp.gsp_candidates(plan))
        assert status == gsp.GSP_ERR_TIMEOUT or limit[1] == 0
        assert status == gsp.GSP_OK or limit[0] < 4_000_000_000
        assert status == gsp.GSP_ERR_TIMEOUT or all(torch.equal(out[i, :n_out], r) for i, r in ref.items())


def test_sub_band_objects_side_by_side(gsp):
    """Objects whose stage 2 needs different amounts of shared memory, used in turn."""
    nchan, nsub, group, n_in = 64, 8, 16, 12000
    x = torch.from_numpy(np.random.default_rng(6).integers(0, 256, (nchan, n_in), dtype=np.uint8)).cuda()
    subs = []
    for step in (4.0, 0.1, 1.0, 8.0):
        d, keep = gsp.make_desc(nchan, 1200.0, 1500.0, 1e-4, n_in, ndm=32, dm_step=step)
        subs.append(gsp.gsp_subband_create(d, nsub, group))
    for sub in subs + subs:
        d1, d2, _ = gsp.gsp_subband_delays(sub)
        n = gsp.gsp_subband_nout(sub, n_in)
        out = torch.full((32, (n + 3) // 4 * 4), -7, dtype=torch.int32, device="cuda")
        gsp.gsp_subband_dedisperse(sub, x, n_in, out)
        gsp.gsp_subband_finish(sub)
        for k in (0, 31):
            ref = torch.zeros(n, dtype=torch.int32, device="cuda")
            for c in range(nchan):
                o = int(d1[k // group, c] + d2[k, c // (nchan // nsub)])
                ref += x[c, o:o + n]
            assert torch.equal(out[k, :n], ref), k


@pytest.mark.parametrize("cycles,starve", [(2_000_000, 1), (1, 0)])
def test_sub_band_waits_that_run_out(gsp, cycles, starve):
    """Stage 2 without copies: a timeout at finish.  Both stages with limits shorter than a copy: a
    timeout or exact sums.  Then exact sums from the same object."""
    nchan, nsub, group, n_in, ndm = 64, 16, 16, 60000, 40
    x = torch.from_numpy(np.random.default_rng(7).integers(0, 256, (nchan, n_in), dtype=np.uint8)).cuda()
    d, keep = gsp.make_desc(nchan, 1200.0, 1500.0, 1e-4, n_in, ndm=ndm, dm_step=1.0)
    sub = gsp.gsp_subband_create(d, nsub, group)
    d1, d2, _ = gsp.gsp_subband_delays(sub)
    n = gsp.gsp_subband_nout(sub, n_in)
    out = torch.full((ndm, (n + 3) // 4 * 4), -7, dtype=torch.int32, device="cuda")
    ref = {}
    for k in (0, 23, ndm - 1):
        at = [int(d1[k // group, c] + d2[k, c // (nchan // nsub)]) for c in range(nchan)]
        ref[k] = sum(x[c, at[c]:at[c] + n].int() for c in range(nchan))
    for limit in [(cycles, starve), (4_000_000_000, 0)] * 3:
        gsp.gsp_subband_set_wait_limit(sub, *limit)
        gsp.gsp_subband_dedisperse(sub, x, n_in, out)
        status = _status(gsp, lambda: gsp.gsp_subband_finish(sub))
        assert status == gsp.GSP_ERR_TIMEOUT or limit[1] == 0
        assert status == gsp.GSP_OK or limit[0] < 4_000_000_000
        assert status == gsp.GSP_ERR_TIMEOUT or all(torch.equal(out[k, :n], r) for k, r in ref.items())
    for bad in [(0, 0), (5_000_000_000, 0), (100, 2)]:
        with pytest.raises(gsp.GspError):
            gsp.gsp_subband_set_wait_limit(sub, *bad)


def test_failed_tuning_leaves_the_plan(gsp, monkeypatch):
    """A plan whose band is split between the two kernels: a tuning call whose launches time out
    changes neither its variant nor the split."""
    monkeypatch.delenv("GSP_DD_VARIANT", raising=False)
    nchan, ndm, n_out = 1024, 240, 50001
    base, _ = gsp.make_desc(nchan, 500.0, 3300.0, 98.304e-6, 1 << 20, ndm=ndm, dm_step=1.0)
    n_in = n_out + int(gsp.gsp_compute_delays(base)[0].max())
    d, keep = gsp.make_desc(nchan, 500.0, 3300.0, 98.304e-6, n_in, ndm=ndm, dm_step=1.0)
    plan = gsp.gsp_plan_create(d, keep)
    x = torch.randint(0, 256, (nchan, (n_in + 15) // 16 * 16), dtype=torch.uint8, device="cuda")
    out = torch.zeros((ndm, (n_out + 3) // 4 * 4), dtype=torch.int32, device="cuda")
    gsp.gsp_dedisperse(plan, x, n_in, out)
    before, want = (gsp.gsp_dedisperse_variants(plan)[1], gsp.gsp_plan_launches(plan)), out.clone()
    assert before[1] == 2
    gsp.gsp_plan_set_wait_limit(plan, 1_000_000, 1)
    assert _status(gsp, lambda: gsp.gsp_plan_tune(plan, x, n_in)) == gsp.GSP_ERR_TIMEOUT
    gsp.gsp_plan_set_wait_limit(plan, 4_000_000_000, 0)
    gsp.gsp_dedisperse(plan, x, n_in, out)
    assert (gsp.gsp_dedisperse_variants(plan)[1], gsp.gsp_plan_launches(plan)) == before
    assert torch.equal(out, want)
    best, _ = gsp.gsp_plan_tune(plan, x, n_in)
    gsp.gsp_dedisperse(plan, x, n_in, out)
    assert gsp.gsp_dedisperse_variants(plan)[1] == best and torch.equal(out, want)


@pytest.mark.parametrize("nchan", [1000, 1023, 1030])
@pytest.mark.parametrize("descending", [False, True])
def test_band_split_in_both_orders(gsp, monkeypatch, nchan, descending):
    """A wide band whose channel count is no whole number of stages is split between the two
    kernels in either channel order, with the same sums as the byte kernel."""
    ndm, n_out = 240, 50001
    base, _ = gsp.make_desc(nchan, 500.0, 3300.0, 98.304e-6, 1 << 20, ndm=ndm, dm_step=1.0)
    n_in = n_out + int(gsp.gsp_compute_delays(base)[0].max())
    g = torch.Generator(device="cuda")
    g.manual_seed(nchan)
    x = torch.randint(0, 256, (nchan, (n_in + 15) // 16 * 16), dtype=torch.uint8, device="cuda", generator=g)
    outs = []
    for variant in (None, "42"):
        if variant:
            monkeypatch.setenv("GSP_DD_VARIANT", variant)
        else:
            monkeypatch.delenv("GSP_DD_VARIANT", raising=False)
        d, keep = gsp.make_desc(nchan, 500.0, 3300.0, 98.304e-6, n_in, ndm=ndm, dm_step=1.0,
                                freq_descending=descending)
        plan = gsp.gsp_plan_create(d, keep)
        outs.append(torch.zeros((ndm, (n_out + 3) // 4 * 4), dtype=torch.int32, device="cuda"))
        gsp.gsp_dedisperse(plan, x, n_in, outs[-1])
        assert gsp.gsp_plan_launches(plan) == (1 if variant else 2)
    assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("block_len", [1 << 20, (1 << 30) + 16, (1 << 31) - 1])
def test_search_blocks_longer_than_the_series(gsp, monkeypatch, block_len):
    """Search blocks up to the longest that a plan accepts, on the tensor-core kernel: no whole
    block, so no candidates, and the same series."""
    monkeypatch.setenv("GSP_DD_VARIANT", str(gsp.gsp_dedisperse_variants()[0] - 1))
    nchan, n_in, ndm = 40, 30000, 20
    d, keep = gsp.make_desc(nchan, 1200.0, 1500.0, 1e-4, n_in, ndm=ndm, dm_step=1.0, block_len=block_len)
    plan = gsp.gsp_plan_create(d, keep)
    x = torch.from_numpy(np.random.default_rng(9).integers(0, 256, (nchan, (n_in + 15) // 16 * 16), dtype=np.uint8)).cuda()
    dl, n_out = gsp.gsp_plan_delays(plan), gsp.gsp_plan_nout(plan, n_in)
    out = torch.zeros((ndm, (n_out + 3) // 4 * 4), dtype=torch.int32, device="cuda")
    gsp.gsp_search(plan, x, n_in, 0, out)
    c, n, st = gsp.gsp_candidates(plan)
    assert n == 0 and st == gsp.GSP_OK
    ref = sum(x[k, int(dl[ndm - 1, k]):int(dl[ndm - 1, k]) + n_out].int() for k in range(nchan))
    assert torch.equal(out[ndm - 1, :n_out], ref)
