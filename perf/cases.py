"""Performance cases: the calls a pulsar-search program makes of this package, through
the public binding (paper_2110_12749_gb300.gsp), over the sizes it is used at.

  listed()             the named cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  what a program holds before the call (inputs, plan, weights)
  run(state)           one pass, returning every output
  work(case)           bytes and operations the pass cannot do without
  exact(case, seed)    the same outputs in 64 bits by plain torch, where they are floats

The kinds, and what each stands for:

  search      gsp_search + gsp_candidates of a filterbank on the device: one beam (or one
              drift-scan chunk) dedispersed and searched, the pipeline's main call.
  dedisperse  gsp_dedisperse into the caller's series, for programs with their own search.
  series      gsp_search_series + gsp_candidates of series that the caller dedispersed.
  host        gsp_search_host: one chunk from pinned host memory to its candidate list.
  batch       gsp_batch_search + gsp_batch_candidates: several beams of different lengths
              and DM grids in one persistent launch.
  subband     gsp_subband_dedisperse: the two-stage sub-band algorithm.
  ddplan      gsp_ddplan_search + gsp_ddplan_candidates: a survey plan whose DM ranges have
              their own step and time downsampling.
  ingest      gsp_ingest_transpose: time-major samples, as files hold them, to channel-major.
  snippets    gsp_ranker_snippets: the 64 x 64 images of one scoring chunk of candidates.
  forward     gsp_ranker_forward: the ranker's logits for one chunk of snippets.
  train       a few gsp_ranker_train_step calls from given weights, then the weights,
              gradients and losses read back.

Inputs follow the synthetic survey data of this repository: 8-bit Gaussian noise around
128, narrowband RFI on a few channels, broadband bursts and dispersed pulses.
"""
import math

import numpy as np
import torch

from paper_2110_12749_gb300 import gsp

# The bands of the repository's workloads: (f_lo, f_hi) in MHz and the sampling time in s.
BANDS = {
    "tiny": (1200.0, 1500.0, 100e-6),
    "crafts": (1000.0, 1500.0, 49.152e-6),
    "wideband": (500.0, 3300.0, 98.304e-6),
    "band1": (271.0, 398.0, 98.304e-6),
}

# Survey plan of the 271-398 MHz band: (low DM, step, trials, downsampling) per range.
BAND1_RANGES = ((0.0, 0.01, 1134, 1), (11.34, 0.03, 362, 2), (22.2, 0.05, 337, 4),
                (39.05, 0.1, 381, 8), (77.15, 0.2, 383, 16), (153.75, 0.5, 380, 32),
                (343.75, 1.0, 344, 64), (687.75, 2.0, 141, 128))

KDM = 4.148808e3  # s MHz^2 / (pc cm^-3)

# Network of the ranker: flat parameter vector w1 b1 w2 b2 w3 b3 w4 b4 w5 b5.
CONVS = ((8, 1), (16, 8), (32, 16))
HIDDEN = 96


def listed():
    return [
        # one small chunk (256 channels, 200 trials): the smallest search, where launches count
        {"name": "search_tiny", "kind": "search", "band": "tiny", "nchan": 256, "n_in": 32768,
         "ndm": 200, "dm_step": 1.0},
        # one full drift-scan beam (4096 channels, 51.5 s, 2000 trials to DM 1000): the benchmark
        {"name": "search_beam", "kind": "search", "band": "crafts", "nchan": 4096,
         "n_in": 1 << 20, "ndm": 2000, "dm_step": 0.5},
        # long sweeps of a wide low band into the caller's series; odd lengths
        {"name": "dedisperse_wideband", "kind": "dedisperse", "band": "wideband", "nchan": 2048,
         "n_in": 600011, "ndm": 3000, "dm_step": 1.0},
        # series dedispersed elsewhere, searched here; a length that is no whole number of blocks
        {"name": "search_series", "kind": "series", "ndm": 500, "n_out": 250001},
        # a chunk as a recorder hands it over, in pinned host memory, to its candidates
        {"name": "search_host", "kind": "host", "band": "crafts", "nchan": 4096, "n_in": 1 << 17,
         "ndm": 2000, "dm_step": 0.5},
        # beams of a multi-beam receiver with their own lengths and DM grids, one launch
        {"name": "batch_beams", "kind": "batch", "band": "crafts", "nchan": 4096,
         "n_in": 196608, "ndm": 1500, "dm_max": 1200.0, "beams": 4},
        # the two-stage algorithm on a chunk of the 4096-channel beam
        {"name": "subband_chunk", "kind": "subband", "band": "crafts", "nchan": 4096,
         "n_in": 1 << 18, "ndm": 2000, "dm_step": 0.5, "nsub": 64, "group": 16},
        # the eight-range survey plan of the 271-398 MHz band, 3462 trials, on 52 s of data
        {"name": "ddplan_band1", "kind": "ddplan", "nchan": 512, "n_in": 1 << 19, "ranges": 8},
        # a chunk of samples in file order, transposed for the search
        {"name": "ingest_chunk", "kind": "ingest", "nchan": 4096, "n_samp": 262144, "pad": 0},
        # one scoring chunk of candidates cut out of a searched chunk's series
        {"name": "snippets_chunk", "kind": "snippets", "ndm": 2000, "n_out": 191852, "n": 4096},
        # the ranker over one scoring chunk
        {"name": "ranker_forward", "kind": "forward", "n": 4096},
        # four training steps at the training batch size
        {"name": "ranker_train", "kind": "train", "n": 256, "steps": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "search", "dedisperse", "dedisperse", "series", "host",
                       "batch", "subband", "ddplan", "ingest", "snippets", "forward", "train"])
    c = {"kind": kind}
    if kind in ("search", "dedisperse", "host"):
        c["band"] = rng.choice(["tiny", "crafts", "crafts", "wideband"])
        if c["band"] == "tiny":
            c["nchan"], c["ndm"] = _log(rng, 64, 1024), _log(rng, 30, 600)
            c["dm_step"] = rng.choice([0.25, 0.5, 1.0])
        elif c["band"] == "crafts":
            c["nchan"], c["ndm"] = _log(rng, 512, 4096), _log(rng, 200, 2500)
            c["dm_step"] = rng.choice([0.25, 0.4, 0.5, 0.6, 0.75])
        else:
            c["nchan"], c["ndm"] = _log(rng, 256, 2048), _log(rng, 100, 3000)
            c["dm_step"] = rng.choice([0.3, 0.5, 1.0])
        f_lo, f_hi, ts = BANDS[c["band"]]
        sweep = KDM * c["dm_step"] * c["ndm"] * (f_lo ** -2 - f_hi ** -2) / ts
        c["n_in"] = int(sweep) + _log(rng, 16384, 262144)
    elif kind == "series":
        c["ndm"], c["n_out"] = _log(rng, 20, 2000), _log(rng, 12000, 300000)
    elif kind == "batch":
        c["band"], c["nchan"] = "crafts", rng.choice([1024, 2048, 4096])
        c["beams"], c["ndm"] = rng.randint(2, 6), rng.randint(1000, 2000)
        c["dm_max"], c["n_in"] = float(rng.randint(500, 1500)), 16 * rng.randint(7000, 14000)
    elif kind == "subband":
        c["band"], c["nchan"] = "crafts", rng.choice([1024, 2048, 4096])
        c["nsub"], c["group"] = rng.choice([16, 32, 64]), rng.choice([8, 12, 16])
        c["ndm"], c["dm_step"] = _log(rng, 300, 2000), rng.choice([0.25, 0.5])
        c["n_in"] = 60000 + _log(rng, 16384, 262144)
    elif kind == "ddplan":
        c["nchan"], c["ranges"] = rng.choice([128, 256, 512]), rng.randint(3, 8)
        c["n_in"] = 340000 + _log(rng, 16384, 400000)
    elif kind == "ingest":
        c["nchan"], c["n_samp"] = _log(rng, 64, 4096), _log(rng, 4096, 1 << 18)
        c["pad"] = rng.choice([0, 0, 4, 16, 3])
    elif kind == "snippets":
        c["ndm"], c["n_out"], c["n"] = _log(rng, 200, 2000), _log(rng, 30000, 191852), _log(rng, 64, 65536)
    elif kind == "forward":
        c["n"] = _log(rng, 16, 4096)
    else:
        c["n"], c["steps"] = _log(rng, 32, 1024), rng.choice([1, 2, 4])
    return c


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _freqs(nchan, f_lo, f_hi):
    return f_lo + (np.arange(nchan) + 0.5) * (f_hi - f_lo) / nchan


def _sweep(nchan, f_lo, f_hi, ts, dm):
    f = _freqs(nchan, f_lo, f_hi)
    return np.floor(KDM * dm * (f ** -2 - f[-1] ** -2) / ts + 0.5).astype(np.int64)


def _filterbank(nchan, n_in, f_lo, f_hi, ts, dm_hi, seed, pulses=12, bursts=3, sigma=20.0):
    """uint8 CUDA [nchan][round16(n_in)]: noise, narrowband RFI, bursts, dispersed pulses."""
    g, r = _gen(seed), np.random.default_rng(seed)
    stride = (n_in + 15) // 16 * 16
    x = torch.empty((nchan, stride), dtype=torch.uint8, device="cuda")
    rows = max(1, (1 << 27) // stride)
    for c in range(0, nchan, rows):
        m = min(rows, nchan - c)
        z = torch.empty((m, stride), device="cuda").normal_(128.0, sigma, generator=g)
        x[c:c + m] = z.round_().clamp_(0, 255).to(torch.uint8)
    del z
    t = torch.arange(stride, device="cuda", dtype=torch.float32)
    for c in r.choice(nchan, max(1, nchan * 30 // 4096), replace=False):
        period, phase = math.exp(r.uniform(math.log(16), math.log(4096))), r.uniform(0, 2 * math.pi)
        s = x[c].float() + 10.0 * sigma * torch.sin(t * (2 * math.pi / period) + phase)
        x[c] = s.round_().clamp_(0, 255).to(torch.uint8)
    for _ in range(bursts):
        w = int(round(math.exp(r.uniform(0, math.log(100)))))
        t0 = int(r.integers(0, max(1, n_in - w)))
        s = x[:, t0:t0 + w].float() + 3.0 * sigma
        x[:, t0:t0 + w] = s.clamp_(0, 255).to(torch.uint8)
    ch = torch.arange(nchan, device="cuda")[:, None]
    for _ in range(pulses):
        dm, w = r.uniform(0.01 * dm_hi, dm_hi), int(round(math.exp(r.uniform(0, math.log(100)))))
        amp = r.uniform(8, 40) * sigma / math.sqrt(nchan * w)
        d = _sweep(nchan, f_lo, f_hi, ts, dm)
        t0 = int(r.integers(0, max(1, n_in - w - int(d.max()))))
        at = (torch.from_numpy(d).cuda()[:, None] + t0 + torch.arange(w, device="cuda")).clamp_(max=n_in - 1)
        noise = torch.rand((nchan, w), device="cuda", generator=g)  # unbiased rounding of amp
        x[ch, at] = (x[ch, at].float() + amp + noise).floor_().clamp_(0, 255).to(torch.uint8)
    return x


def _series(ndm, n_out, seed):
    """int32 CUDA [ndm][round4(n_out)]: dedispersed-like series (4096 channels of noise) with
    slow drifts, a few loud blocks and boxcar pulses that spread over neighbouring trials."""
    g, r = _gen(seed), np.random.default_rng(seed)
    stride = (n_out + 3) // 4 * 4
    D = torch.empty((ndm, stride), dtype=torch.int32, device="cuda")
    t = torch.arange(stride, device="cuda", dtype=torch.float32)
    drift = 400.0 * torch.sin(t * (2 * math.pi / 5000.0)) + 300.0 * torch.sin(t * (2 * math.pi / 37000.0))
    rows = max(1, (1 << 26) // stride)
    for d in range(0, ndm, rows):
        m = min(rows, ndm - d)
        z = torch.empty((m, stride), device="cuda").normal_(524288.0, 1280.0, generator=g)
        D[d:d + m] = (z + drift).round_().to(torch.int32)
    for _ in range(2):
        t0 = int(r.integers(0, max(1, n_out - 600)))
        D[:, t0:t0 + 600] += (torch.arange(600, device="cuda", dtype=torch.int32) % 7) * 4000
    for _ in range(40):
        w, d0 = int(round(math.exp(r.uniform(0, math.log(150))))), int(r.integers(0, ndm))
        t0 = int(r.integers(0, max(1, n_out - w - 64)))
        amp = r.uniform(7, 40) * 1280.0 / math.sqrt(w)
        for k in range(max(0, d0 - 6), min(ndm, d0 + 7)):
            D[k, t0 + abs(k - d0):t0 + abs(k - d0) + w] += int(amp * (1 - abs(k - d0) / 8))
    return D


def _cands(case, seed):
    """Candidate records spread as a search leaves them (time, DM and widths)."""
    r = np.random.default_rng(seed + 7)
    n, Ls = case["n"], case["n_out"] // 1024 * 1024
    c = np.zeros(n, gsp.CAND_DTYPE)
    c["dm_idx"] = np.sort(r.integers(0, case["ndm"], n))
    c["t"] = r.integers(0, Ls - 150, n)
    c["width"] = r.choice(gsp.DEFAULT_WIDTHS, n, p=np.array([3, 2, 2, 2, 3, 4, 6, 8, 10, 14, 18, 24, 30]) / 126)
    c["snr"] = r.uniform(6, 12, n)
    return c


def _create(make, nchan, f_lo, f_hi, ts, n_in, ndm, dm_step):
    """make(desc) on a DM grid from 0; a grid with a delay on a rounding tie, which plans
    refuse, is moved by a little, as a program would."""
    for k in range(8):
        desc, keep = gsp.make_desc(nchan, f_lo, f_hi, ts, n_in, ndm=ndm, dm_lo=1e-4 * k,
                                   dm_step=dm_step)
        try:
            return make(desc, keep)
        except gsp.GspError as e:
            if e.status != gsp.GSP_ERR_TIE:
                raise
    raise RuntimeError("no tie-free DM grid")


def _plan(case):
    f_lo, f_hi, ts = BANDS[case["band"]]
    return _create(gsp.gsp_plan_create, case["nchan"], f_lo, f_hi, ts, case["n_in"], case["ndm"],
                   case["dm_step"])


def _images(n, seed):
    """FP32 [n][64][64] snippets: unit noise, half of them with a bow-tie pulse."""
    g, r = _gen(seed), np.random.default_rng(seed)
    x = torch.empty((n, 64, 64), device="cuda").normal_(0, 1, generator=g)
    y = torch.from_numpy(r.integers(0, 2, n).astype(np.int32)).cuda()
    row = torch.arange(64, device="cuda", dtype=torch.float32)
    off = (row[:, None] - 32).abs()
    shape = torch.exp(-((row[None, :] - 32) / (1.5 + 0.4 * off)) ** 2) * torch.exp(-off / 12)
    amp = torch.from_numpy(r.uniform(2, 8, n).astype(np.float32)).cuda()
    return x + (amp * y)[:, None, None] * shape, y


def _params(seed):
    """He-uniform weights, zero biases, in the ranker's flat order."""
    r = np.random.default_rng(seed + 11)
    out = []
    for co, ci in CONVS:
        out += [r.uniform(-1, 1, co * ci * 9) * math.sqrt(6.0 / (ci * 9)), np.zeros(co)]
    out += [r.uniform(-1, 1, HIDDEN * 2048) * math.sqrt(6.0 / 2048), np.zeros(HIDDEN)]
    out += [r.uniform(-1, 1, 2 * HIDDEN) * math.sqrt(6.0 / HIDDEN), np.zeros(2)]
    return np.concatenate(out).astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    if kind in ("search", "dedisperse", "host"):
        f_lo, f_hi, ts = BANDS[case["band"]]
        s["plan"] = _plan(case)
        x = _filterbank(case["nchan"], case["n_in"], f_lo, f_hi, ts,
                        case["dm_step"] * case["ndm"], seed)
        s["slots"] = _slots(case["ndm"], gsp.gsp_plan_nout(s["plan"], case["n_in"]))
        if kind == "host":
            s["x"] = torch.empty(x.shape, dtype=torch.uint8, pin_memory=True)
            s["x"].copy_(x)
        else:
            s["x"] = x
        if kind == "dedisperse":
            n_out = gsp.gsp_plan_nout(s["plan"], case["n_in"])
            s["D"] = torch.zeros((case["ndm"], (n_out + 3) // 4 * 4), dtype=torch.int32, device="cuda")
            s["n_out"] = n_out
    elif kind == "series":
        desc, keep = gsp.make_desc(64, 1200.0, 1500.0, 1e-4, case["n_out"], ndm=case["ndm"],
                                   dm_lo=0.0, dm_step=0.0)
        s["plan"] = gsp.gsp_plan_create(desc, keep)
        s["D"] = _series(case["ndm"], case["n_out"], seed)
        s["slots"] = _slots(case["ndm"], case["n_out"])
    elif kind == "batch":
        f_lo, f_hi, ts = BANDS[case["band"]]
        plans, xs, n_ins = [], [], []
        for b in range(case["beams"]):
            ndm = case["ndm"] - 101 * b                # beams with their own grids and lengths
            dm_max = case["dm_max"] * (1.0 - 0.1 * b)
            n_in = case["n_in"] - 8208 * b
            plans.append(_create(gsp.gsp_plan_create, case["nchan"], f_lo, f_hi, ts, n_in, ndm,
                                 dm_max / ndm))
            xs.append(_filterbank(case["nchan"], n_in, f_lo, f_hi, ts, dm_max, seed + 1000 * b))
            n_ins.append(n_in)
        s["batch"] = gsp.gsp_batch_create(plans, gsp.GSP_BATCH_PERSISTENT)
        s["xs"], s["n_ins"] = xs, n_ins
        s["slots"] = sum(_slots(p.ndm, gsp.gsp_plan_nout(p, n)) for p, n in zip(plans, n_ins))
    elif kind == "subband":
        f_lo, f_hi, ts = BANDS[case["band"]]
        s["sub"] = _create(lambda d, keep: gsp.gsp_subband_create(d, case["nsub"], case["group"]),
                           case["nchan"], f_lo, f_hi, ts, case["n_in"], case["ndm"], case["dm_step"])
        s["x"] = _filterbank(case["nchan"], case["n_in"], f_lo, f_hi, ts,
                             case["dm_step"] * case["ndm"], seed)
        s["n_out"] = gsp.gsp_subband_nout(s["sub"], case["n_in"])
        s["D"] = torch.zeros((case["ndm"], (s["n_out"] + 3) // 4 * 4), dtype=torch.int32, device="cuda")
    elif kind == "ddplan":
        f_lo, f_hi, ts = BANDS["band1"]
        ranges = BAND1_RANGES[:case["ranges"]]
        desc, keep = gsp.make_desc(case["nchan"], f_lo, f_hi, ts, case["n_in"], ndm=1)
        s["keep"] = keep
        s["dd"] = gsp.gsp_ddplan_create(desc, ranges)
        s["x"] = _filterbank(case["nchan"], case["n_in"], f_lo, f_hi, ts, 60.0, seed)
        s["slots"] = sum(_slots(r[2], case["n_in"] // r[3]) for r in ranges)
    elif kind == "ingest":
        C, N = case["nchan"], case["n_samp"]
        s["x"] = torch.randint(0, 256, (N, C + case["pad"]), dtype=torch.uint8, device="cuda",
                               generator=_gen(seed))
        s["out"] = torch.zeros((C, (N + 15) // 16 * 16), dtype=torch.uint8, device="cuda")
    elif kind == "snippets":
        desc, keep = gsp.make_desc(4096, 1000.0, 1500.0, 49.152e-6, case["n_out"], ndm=case["ndm"],
                                   dm_lo=0.0, dm_step=0.0)
        s["plan"] = gsp.gsp_plan_create(desc, keep)
        s["D"] = _series(case["ndm"], case["n_out"], seed)
        gsp.gsp_search_series(s["plan"], s["D"], case["n_out"])
        s["cands"] = torch.from_numpy(_cands(case, seed).view(np.uint8).copy()).cuda()
        s["out"] = torch.zeros((case["n"], 64, 64), device="cuda")
    elif kind == "forward":
        s["ranker"] = gsp.gsp_ranker_create(4096)
        gsp.gsp_ranker_set_params(s["ranker"], _params(seed))
        s["x"], _ = _images(case["n"], seed)
        s["logits"] = torch.zeros((case["n"], 2), device="cuda")
    else:
        s["ranker"] = gsp.gsp_ranker_create(case["n"])
        s["params"] = _params(seed)
        x, y = _images(case["n"] * case["steps"], seed)
        s["x"] = x.reshape(case["steps"], case["n"], 64, 64)
        s["y"] = y.reshape(case["steps"], case["n"])
        s["loss"] = torch.zeros(case["steps"], device="cuda")
    return s


# ------------------------------------------------------------------ one pass

def _table(c, n, rows):
    """The candidate list as the fixed-size columns that a program stores (empty past the
    end); rows: one per DM trial and search window, the most there can be."""
    out = {"n": int(n)}
    for name in ("dm_idx", "width", "t", "beam", "snr"):
        out[name] = np.zeros(rows, c.dtype[name])
        out[name][:c.size] = c[name]
    return out


def _slots(ndm, n_out):
    return min(1 << 20, ndm * (n_out // 1024 + 1))


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "search":
        gsp.gsp_search(s["plan"], s["x"], case["n_in"])
        c, n, _ = gsp.gsp_candidates(s["plan"])
        return _table(c, n, s["slots"])
    if kind == "dedisperse":
        gsp.gsp_dedisperse(s["plan"], s["x"], case["n_in"], s["D"])
        return s["D"][:, :s["n_out"]]
    if kind == "series":
        gsp.gsp_search_series(s["plan"], s["D"], case["n_out"])
        c, n, _ = gsp.gsp_candidates(s["plan"])
        return _table(c, n, s["slots"])
    if kind == "host":
        c, n, _ = gsp.gsp_search_host(s["plan"], s["x"], case["n_in"])
        return _table(c, n, s["slots"])
    if kind == "batch":
        gsp.gsp_batch_search(s["batch"], s["xs"], s["n_ins"])
        c, n, _ = gsp.gsp_batch_candidates(s["batch"])
        return _table(c, n, s["slots"])
    if kind == "subband":
        gsp.gsp_subband_dedisperse(s["sub"], s["x"], case["n_in"], s["D"])
        return s["D"][:, :s["n_out"]]
    if kind == "ddplan":
        gsp.gsp_ddplan_search(s["dd"], s["x"], case["n_in"])
        c, n, _ = gsp.gsp_ddplan_candidates(s["dd"])
        return _table(c, n, s["slots"])
    if kind == "ingest":
        gsp.gsp_ingest_transpose(s["x"], case["n_samp"], case["nchan"], s["out"])
        return s["out"][:, :case["n_samp"]]
    if kind == "snippets":
        gsp.gsp_ranker_snippets(s["plan"], s["D"], s["cands"], s["out"])
        return s["out"]
    if kind == "forward":
        gsp.gsp_ranker_forward(s["ranker"], s["x"], case["n"], s["logits"])
        return s["logits"]
    gsp.gsp_ranker_set_params(s["ranker"], s["params"])
    for k in range(case["steps"]):
        gsp.gsp_ranker_train_step(s["ranker"], s["x"][k], s["y"][k], case["n"], 1e-3,
                                  s["loss"][k:k + 1])
    p, g = gsp.gsp_ranker_get_params(s["ranker"])
    return {"params": p, "grads": g, "loss": s["loss"]}


# ------------------------------------------------------------------ work

def _nout(band, nchan, n_in, dm_hi):
    f_lo, f_hi, ts = BANDS[band]
    return max(0, n_in - int(_sweep(nchan, f_lo, f_hi, ts, dm_hi)[0]))


def _search_ops(ndm, n_out):
    return ndm * n_out * len(gsp.DEFAULT_WIDTHS) * 4  # per width: sum, trend, scale, maximum


def work(case):
    kind = case["kind"]
    if kind in ("search", "dedisperse", "host"):
        n_out = _nout(case["band"], case["nchan"], case["n_in"], case["dm_step"] * (case["ndm"] - 1))
        adds = case["nchan"] * case["ndm"] * n_out
        nbytes = case["nchan"] * case["n_in"]
        if kind == "dedisperse":
            return {"bytes": nbytes + 4 * case["ndm"] * n_out, "flops": adds}
        return {"bytes": nbytes, "flops": adds + _search_ops(case["ndm"], n_out)}
    if kind == "series":
        return {"bytes": 4 * case["ndm"] * case["n_out"], "flops": _search_ops(case["ndm"], case["n_out"])}
    if kind == "batch":
        nbytes = ops = 0
        for b in range(case["beams"]):
            ndm, dm_max, n_in = case["ndm"] - 101 * b, case["dm_max"] * (1 - 0.1 * b), case["n_in"] - 8208 * b
            n_out = _nout(case["band"], case["nchan"], n_in, dm_max * (ndm - 1) / ndm)
            nbytes += case["nchan"] * n_in
            ops += case["nchan"] * ndm * n_out + _search_ops(ndm, n_out)
        return {"bytes": nbytes, "flops": ops}
    if kind == "subband":
        n_out = _nout(case["band"], case["nchan"], case["n_in"], case["dm_step"] * (case["ndm"] - 1))
        nsdm = (case["ndm"] + case["group"] - 1) // case["group"]
        return {"bytes": case["nchan"] * case["n_in"] + 4 * case["ndm"] * n_out,
                "flops": (nsdm * case["nchan"] + case["ndm"] * case["nsub"]) * n_out}
    if kind == "ddplan":
        ops = 0
        for lo, step, ndm, ds in BAND1_RANGES[:case["ranges"]]:
            n_out = _nout("band1", case["nchan"], case["n_in"], lo + step * (ndm - 1)) // ds
            ops += case["nchan"] * ndm * n_out + _search_ops(ndm, n_out)
        return {"bytes": case["nchan"] * case["n_in"], "flops": ops}
    if kind == "ingest":
        return {"bytes": 2 * case["nchan"] * case["n_samp"], "flops": 0}
    if kind == "snippets":
        n = case["n"]
        # the images written, and the samples under them read (at most the whole series)
        return {"bytes": n * 64 * 64 * 4 + min(n * 64 * 64 * 16, case["ndm"] * case["n_out"]) * 4,
                "flops": n * 64 * 64 * 16}
    per = 2 * (64 * 64 * 8 * 9 + 32 * 32 * 16 * 72 + 16 * 16 * 32 * 144 + 2048 * HIDDEN + 2 * HIDDEN)
    if kind == "forward":
        return {"bytes": case["n"] * (64 * 64 * 4 + 8) + 202786 * 4, "flops": case["n"] * per}
    return {"bytes": case["steps"] * (case["n"] * 64 * 64 * 4 + 202786 * 4 * 7),
            "flops": case["steps"] * case["n"] * 3 * per}


# ------------------------------------------------------------------ 64-bit values

def _exact_snippets(case, seed):
    D, c, B = _series(case["ndm"], case["n_out"], seed), _cands(case, seed), 1024
    nb = case["n_out"] // B
    Ls = nb * B
    r = D[:, :Ls].double().reshape(case["ndm"], nb, B)
    j = torch.arange(B, device="cuda", dtype=torch.float64) - (B - 1) / 2
    r -= r.mean(2, keepdim=True)
    r -= ((r * j).sum(2, keepdim=True) / (j * j).sum()) * j
    sig = r.square().mean(2).sqrt()
    ref = sig.sort(1).values[:, (nb - 1) // 2]
    bad = (sig < 0.5 * ref[:, None]) | (sig > 2.5 * ref[:, None])
    r[bad] = 0.0
    r /= ref[:, None, None]
    P = torch.zeros((case["ndm"], Ls + 1), dtype=torch.float64, device="cuda")
    torch.cumsum(r.reshape(case["ndm"], Ls), 1, out=P[:, 1:])
    del r, D
    out = torch.zeros((case["n"], 64, 64), dtype=torch.float64, device="cuda")
    k = torch.arange(64, device="cuda")
    for a in range(0, case["n"], 4096):
        d = torch.from_numpy(c["dm_idx"][a:a + 4096].astype(np.int64)).cuda()
        t = torch.from_numpy(c["t"][a:a + 4096].copy()).cuda()
        w = torch.from_numpy(c["width"][a:a + 4096].astype(np.int64)).cuda()
        f = (w // 4).clamp(min=1)
        lo = (t + w // 2 - 32 * f)[:, None] + k * f[:, None]
        row = d[:, None] - 32 + k
        ok = (row >= 0) & (row < case["ndm"])
        row = row.clamp(0, case["ndm"] - 1)[:, :, None]
        v = P[row, (lo + f[:, None]).clamp(0, Ls)[:, None, :]] - P[row, lo.clamp(0, Ls)[:, None, :]]
        out[a:a + 4096] = v * ok[:, :, None] / f.double().sqrt()[:, None, None]
    return out


def _network(p, x):
    F, h, at = torch.nn.functional, x[:, None], 0
    for co, ci in CONVS:
        w = p[at:at + co * ci * 9].reshape(co, ci, 3, 3)
        b = p[at + co * ci * 9:at + co * ci * 9 + co]
        at += co * ci * 9 + co
        h = F.max_pool2d(F.conv2d(h, w, b, padding=1).relu(), 2)
    h = h.permute(0, 2, 3, 1).reshape(x.shape[0], 2048)
    w, b = p[at:at + HIDDEN * 2048].reshape(HIDDEN, 2048), p[at + HIDDEN * 2048:at + HIDDEN * 2049]
    at += HIDDEN * 2049
    h = (h @ w.T + b).relu()
    return h @ p[at:at + 2 * HIDDEN].reshape(2, HIDDEN).T + p[at + 2 * HIDDEN:]


def exact(case, seed):
    kind = case["kind"]
    if kind == "snippets":
        return _exact_snippets(case, seed)
    if kind == "forward":
        x, _ = _images(case["n"], seed)
        p = torch.from_numpy(_params(seed)).cuda().double()
        return torch.cat([_network(p, x[a:a + 256].double()) for a in range(0, case["n"], 256)])
    if kind == "train":
        x, y = _images(case["n"] * case["steps"], seed)
        p = torch.from_numpy(_params(seed)).cuda().double()
        m, v, losses = torch.zeros_like(p), torch.zeros_like(p), []
        for k in range(case["steps"]):
            q, n = p.clone().requires_grad_(True), case["n"]
            loss = torch.nn.functional.cross_entropy(_network(q, x[k * n:(k + 1) * n].double()),
                                                     y[k * n:(k + 1) * n].long())
            loss.backward()
            g = q.grad
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            p = p - 1e-3 * (m / (1 - 0.9 ** (k + 1))) / ((v / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
            losses.append(loss.detach())
        return {"params": p, "grads": g, "loss": torch.stack(losses)}
    # series, transposed bytes and candidate lists are whole numbers (and the length of a list
    # is decided by them): there is nothing to compare in 64 bits
    return None
