"""The tensor-core dedispersion kernel against the CPU oracle, bit-exact, where it
can go wrong: channel counts around its chunks of 8, a single DM trial and partial
DM blocks, output lengths around its tiles, unsorted and steep DM grids (several row
moves between two channels), both channel orders, padded strides, saturated input,
and search blocks of one and several per tile (fused block sums)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MMA_VARIANT = 45

# (nchan, DM grid, n_out, descending, input and output padding, block length, saturated)
CASES = [
    (1, np.arange(3.0), 17, False, 0, 1024, False),
    (7, np.arange(16.0), 1, False, 16, 1024, False),
    (8, np.arange(17.0), 2047, True, 0, 1024, False),
    (9, np.arange(1.0), 2049, False, 32, 1024, False),
    (65, np.linspace(0.0, 40.0, 33), 4100, True, 16, 1024, False),
    (300, np.linspace(0.0, 400.0, 20), 3000, False, 0, 1500, False),      # too steep: byte kernel
    (300, np.linspace(0.0, 150.0, 20), 3000, False, 0, 1500, False),      # steep: repeated moves
    (130, np.array([9.0, 2.0, 30.0, 4.0, 4.0, 55.0, 0.0]), 5000, False, 16, 1024, False),
    (512, np.linspace(0.0, 20.0, 48), 9000, False, 0, 4096, True),
]


@pytest.fixture(scope="module")
def gsp():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2110_12749_gb300 import build, gsp as g
    build.build()
    g.lib()
    return g


@pytest.mark.parametrize("case", range(len(CASES)))
def test_tensor_core_dedispersion_bit_exact(gsp, orc, monkeypatch, case):
    nchan, dms, n_out, desc_order, pad, block, sat = CASES[case]
    rng = np.random.default_rng(case)
    dl, _ = orc.delays(nchan, 1200.0, 1500.0, 1e-4, dms)   # ascending channels
    if desc_order:
        dl = np.ascontiguousarray(dl[:, ::-1])
    n_in = n_out + orc.max_delay(dl)
    stride = (n_in + 15) // 16 * 16 + pad
    x = np.full((nchan, stride), 255, np.uint8) if sat else \
        rng.integers(0, 256, (nchan, stride), dtype=np.uint8)
    ref = orc.dedisperse(x, n_in, dl)
    monkeypatch.setenv("GSP_DD_VARIANT", str(MMA_VARIANT))
    d, keep = gsp.make_desc(nchan, 1200.0, 1500.0, 1e-4, n_in, dms=dms, block_len=block,
                            window_len=1024, threshold=4.0, freq_descending=desc_order)
    plan = gsp.gsp_plan_create(d, keep)
    used = gsp.gsp_dedisperse_variants(plan)[1]
    # 16 neighbouring trials have to fit a tile of 2048 samples
    spread = max((dl[min(b + 15, len(dms) - 1)] - dl[b]).max() for b in range(0, len(dms), 16))
    assert used == MMA_VARIANT if spread < 1900 else used >= 0
    xd = torch.from_numpy(x).cuda()
    out = torch.full((len(dms), (n_out + 3) // 4 * 4 + pad), -7, dtype=torch.int32, device="cuda")
    gsp.gsp_dedisperse(plan, xd, n_in, out)
    o = out.cpu().numpy()
    assert (o[:, :n_out].astype(np.int64) == ref).all()
    assert (o[:, n_out:] == -7).all()
    # fused block sums: the same statistics and candidates as a search of the series
    gsp.gsp_search(plan, xd, n_in)
    c1, n1, _ = gsp.gsp_candidates(plan)
    s1 = gsp.gsp_search_stats(plan, n_out)
    gsp.gsp_search_series(plan, out, n_out)
    c2, n2, _ = gsp.gsp_candidates(plan)
    s2 = gsp.gsp_search_stats(plan, n_out)
    assert n1 == n2 and (c1 == c2).all()
    assert (s1["sigma_b"] == s2["sigma_b"]).all() and (s1["bad"] == s2["bad"]).all()


def test_plan_chooses_by_grid(gsp, monkeypatch):
    """Fine DM grids of a narrow band take the tensor-core kernel, a wide low band does not."""
    monkeypatch.delenv("GSP_DD_VARIANT", raising=False)
    for lo, hi, ts, step, n, mma in [(1000.0, 1500.0, 49.152e-6, 0.5, 64, True),
                                     (500.0, 3300.0, 98.304e-6, 20.0, 64, False)]:
        d, keep = gsp.make_desc(1024, lo, hi, ts, 1 << 19, ndm=n, dm_step=step)
        used = gsp.gsp_dedisperse_variants(gsp.gsp_plan_create(d, keep))[1]
        assert (used == MMA_VARIANT) == mma
