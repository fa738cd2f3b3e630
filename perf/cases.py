"""The work that users of this library have it do, as measurable cases.

Every case goes through the public entry points (search.Plan and the af_* calls
of _lib).  Sizes are those of the repository's own workloads, tests and
benchmark: the 256-channel check search, the 4096-channel full-band search,
the multi-beam survey's 1024-channel beams, and the classifier's batches.
Inputs are synthetic, drawn on the GPU from the seed alone: 8-bit noise with
dispersed pulses, DM-time planes of such data, and min-max normalised 64 x 64
cut-outs.  exact() restates each step in 64 bits with plain torch.
"""
import json
import math
import os

import numpy as np
import torch

from paper_2511_02328_gb300 import _lib, synth
from paper_2511_02328_gb300.search import Plan

F_LO, F_HI = 1000.0, 1500.0
K_DM = 4.148808e3
CKPT = os.path.join("paper_2511_02328_gb300", "data", "stream_cnn_4096ch.ckpt")
CH = (2, 16, 32, 64)
CAP = 1 << 14  # candidates kept of a search
SIZES = (("w0", (16, 3, 3, 2)), ("b0", (16,)), ("w1", (32, 3, 3, 16)), ("b1", (32,)), ("w2", (64, 3, 3, 32)),
         ("b2", (64,)), ("fw", (2, 64)), ("fb", (2,)))


def listed():
    return [
        # one beam's short chunk, searched on the device: the check workload; launches and latency count
        dict(name="search_256ch", kind="search", nchan=256, nsamp=1 << 15, ndm=501, dm_step=1.0, tsamp_us=98.304,
             wmax=32),
        # the full-band search, the benchmark's step: dedispersion, boxcar S/N and candidates of a resident chunk
        dict(name="search_4096ch", kind="search", nchan=4096, nsamp=1 << 18, ndm=1001, dm_step=1.0, tsamp_us=49.152,
             wmax=256),
        # a survey beam from pinned host memory to a candidate list: the one-call search with its copies
        dict(name="host_1024ch", kind="host", nchan=1024, nsamp=1 << 17, ndm=1001, dm_step=1.0, tsamp_us=196.608,
             wmax=256),
        # two beams of a stream, a hop of new samples each: search, clustering and classification of each window
        dict(name="stream_1024ch", kind="stream", nchan=1024, nsamp=1 << 16, ndm=501, dm_step=2.0, tsamp_us=196.608,
             wmax=64),
        # the paper's two-stage subband scheme on the full-band chunk (approximate, for larger DM counts)
        dict(name="subband_4096ch", kind="subband", nchan=4096, nsamp=1 << 18, ndm=1001, dm_step=1.0,
             tsamp_us=49.152, n0=8, nsub=64),
        # cleaning and reducing a full-band chunk before the search: zero-DM filter, then downsampling by 8
        dict(name="prep_4096ch", kind="prep", nchan=4096, nsamp=1 << 18, factor=8),
        # median / MAD row statistics and the robust S/N of a full-band plane (its rows are ragged: 215,261 samples)
        dict(name="robust_1001dm", kind="robust", ndm=1001, nout=215261, nchan=4096, wmax=256),
        # the same plane cut into 0.5 s slices and rendered as 512 x 512 images for a detector
        dict(name="grid_1001dm", kind="grid", ndm=1001, nout=215261, nchan=4096, ns=10173, m=512),
        # cut-outs of a dense window's 256 candidates and their classification
        dict(name="classify_256", kind="classify", nchan=4096, nsamp=1 << 16, ndm=401, dm_step=1.0, tsamp_us=98.304,
             n=256),
        # classifying the few clusters of one streamed window: the smallest call
        dict(name="infer_16", kind="infer", n=16),
        # an epoch of 2048 samples in the training script's batches of 256
        dict(name="train_256", kind="train", n=256, steps=8),
        # one step on a large batch
        dict(name="train_4096", kind="train", n=4096, steps=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "host", "stream", "subband", "prep", "robust", "grid", "classify",
                       "infer", "train"])
    if kind in ("search", "host", "stream", "subband"):
        # the band's time resolution follows the channel count; the largest delay leaves over half of the chunk
        lo, hi = {"search": (100, 4096), "host": (128, 2048), "stream": (128, 1024), "subband": (512, 4096)}[kind]
        nchan = _log(rng, lo, hi)
        if kind == "stream":
            nchan = max(2, nchan // 64) * 64
        nsamp = _log(rng, 1 << 14, 1 << 17)
        if rng.random() < 0.6:
            nsamp = max(nsamp // 64, 256) * 64
        step = rng.choice([0.5, 1.0, 2.0])
        ndm = max(40, min(_log(rng, 64, 1500), int(1.2e11 / (nchan * nsamp))))
        tsamp = 49.152 * max(1, 4096 // nchan)
        while ndm * step * 2.305 / 1000.0 / (tsamp * 1e-6) > 0.45 * nsamp:
            tsamp *= 2
        c = dict(kind=kind, nchan=nchan, nsamp=nsamp, ndm=ndm, dm_step=step, tsamp_us=tsamp)
        if kind == "subband":
            return dict(c, n0=rng.choice([4, 8, 16]), nsub=rng.choice([32, 64, 128]))
        return dict(c, wmax=rng.choice([16, 32, 64, 128, 256]))
    if kind == "prep":
        nsamp = _log(rng, 1 << 14, 1 << 18)
        if rng.random() < 0.5:
            nsamp = nsamp // 64 * 64
        return dict(kind=kind, nchan=_log(rng, 64, 4096), nsamp=nsamp, factor=rng.choice([2, 3, 4, 5, 8, 10, 16, 32]))
    if kind in ("robust", "grid"):
        ndm, nout = _log(rng, 64, 2001), _log(rng, 10000, 215261)
        ndm = min(ndm, int(2.2e8 / nout))
        c = dict(kind=kind, ndm=ndm, nout=nout, nchan=rng.choice([256, 1024, 2048, 4096]))
        if kind == "robust":
            return dict(c, wmax=rng.choice([16, 32, 64, 128, 256]))
        return dict(c, ns=rng.randint(2000, min(10173, nout)), m=rng.choice([256, 512]))
    if kind == "classify":
        return dict(kind=kind, nchan=64 * rng.randint(4, 64), nsamp=16 * _log(rng, 1536, 4096),
                    ndm=rng.randint(101, 401), dm_step=1.0, tsamp_us=98.304, n=_log(rng, 8, 256))
    if kind == "infer":
        return dict(kind=kind, n=_log(rng, 1, 4096))
    n = _log(rng, 64, 4096)
    return dict(kind=kind, n=n, steps=8 if n <= 512 else 1)


# ---- inputs ---------------------------------------------------------------

def _delays(c):
    """Delay table [ndm][nchan] (int64): round half away from zero of K DM / tsamp (1/fc^2 - 1/fref^2)."""
    f = F_LO + (np.arange(c["nchan"]) + 0.5) * (F_HI - F_LO) / c["nchan"]
    a = K_DM * _dms(c) / (c["tsamp_us"] * 1e-6)
    b = 1.0 / (f * f) - 1.0 / (F_HI * F_HI)
    return np.floor(a[:, None] * b[None, :] + 0.5).astype(np.int64)


def _dms(c):
    return np.arange(c["ndm"], dtype=np.float64) * c["dm_step"]


def _widths(c):
    return [1 << k for k in range(c["wmax"].bit_length()) if 1 << k <= c["wmax"]]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _filterbank(c, seed, hop=None):
    """8-bit noise with five dispersed pulses over the chunk, S/N 12 to 30; with hop, that many samples
    of a stream which repeats them (pulses that pass its end go on at its beginning)."""
    nsamp = hop or c["nsamp"]
    rng = np.random.default_rng(seed)
    dms = _dms(c)
    pulses = []
    for k in range(5):
        dm = float(rng.uniform(0.1, 0.9) * dms[-1])
        one = dict(c, ndm=2, dm_step=dm)
        off = _delays(one)[1]
        t0 = int((k + rng.uniform(0.2, 0.6)) * (hop or nsamp - off.max()) / 5)
        off = (off + t0) % nsamp
        w = int(2 ** rng.uniform(0, 5))
        pulses.append(synth.Pulse(off, w, synth.pulse_amplitude(rng.uniform(12.0, 30.0), c["nchan"], w)))
    return synth.filterbank_torch(c["nchan"], nsamp, seed, pulses=pulses)


def _plane(c, seed):
    """A DM-time plane of noise (sums of nchan 8-bit samples) with a few wide pulses on neighbouring rows."""
    g, rng = _gen(seed), np.random.default_rng(seed)
    y = torch.empty((c["ndm"], c["nout"]), dtype=torch.int32, device="cuda")
    sigma = 12.0 * math.sqrt(c["nchan"])
    for d0 in range(0, c["ndm"], 256):
        z = torch.randn(y[d0:d0 + 256].shape, generator=g, device="cuda")
        y[d0:d0 + 256] = (z * sigma + 128.0 * c["nchan"]).round_().int()
    for _ in range(20):
        d, t, w = int(rng.integers(0, c["ndm"])), int(rng.integers(0, c["nout"] - 64)), int(rng.integers(1, 64))
        y[max(0, d - 5):d + 6, t:t + w] += int(8 * sigma / math.sqrt(w))
    return y


def _images(n, seed):
    """Cut-outs as the classifier sees them: min-max normalised noise, half of them with a bright column."""
    g = _gen(seed)
    z = torch.randn((n, 64, 64, 2), generator=g, device="cuda")
    y = torch.randint(0, 2, (n,), generator=g, device="cuda", dtype=torch.int32)
    z[:, :, 31:33] += 3.0 * y[:, None, None, None]
    lo, hi = z.amin(dim=(1, 2), keepdim=True), z.amax(dim=(1, 2), keepdim=True)
    return ((z - lo) / (hi - lo + 1e-6)).to(torch.bfloat16), y


def _initial(seed):
    """He-normal weights, zero biases, in the library's flat order."""
    rng = np.random.default_rng(seed)
    out = []
    for name, shape in SIZES:
        k = int(np.prod(shape))
        sd = {"w": math.sqrt(2.0 / (k // shape[0])), "f": 0.125, "b": 0.0}[name[0]] if name != "fb" else 0.0
        out.append(rng.normal(0.0, 1.0, k) * sd)
    return np.concatenate(out).astype(np.float32)


def _trained():
    """The shipped checkpoint's parameters: a JSON header line, then little-endian fp32."""
    with open(CKPT, "rb") as f:
        json.loads(f.readline())
        return np.frombuffer(f.read(4 * sum(int(np.prod(s)) for _, s in SIZES)), dtype="<f4").copy()


def _candidates(c, nout, seed):
    rng = np.random.default_rng(seed + 17)
    a = np.zeros(c["n"], dtype=_lib.CAND_DTYPE)
    a["dm_idx"] = rng.integers(0, c["ndm"], c["n"])
    a["t"] = rng.integers(0, nout, c["n"])
    a["width"] = 2 ** rng.integers(0, 9, c["n"])
    a["abs_sample"] = a["t"]
    return a


class _Handle:
    """A library handle that is given back with the state that holds it."""

    def __init__(self, h, close):
        self.h, self._close = h, close

    def __del__(self):
        try:
            self._close(self.h)
        except Exception:
            pass


def _model(max_batch, params):
    m = _Handle(_lib.af_model_create(max_batch, 1), _lib.af_model_destroy)
    _lib.af_model_set_params(m.h, params)
    return m


def prepare(case, seed):
    c = dict(case)
    k = c["kind"]
    s = dict(c)
    dev = "cuda"
    if k in ("search", "host", "subband", "classify"):
        tsamp = c["tsamp_us"] * 1e-6
        sub = dict(n0=c["n0"], nsub=c["nsub"]) if k == "subband" else None
        p = s["plan"] = Plan(c["nchan"], F_LO, F_HI, tsamp, _dms(c), subband=sub)
        nout = s["nout"] = p.nout(c["nsamp"])
        x = _filterbank(c, seed)
        if k == "host":
            s["h"] = torch.empty(x.shape, dtype=torch.uint8, pin_memory=True)
            s["h"].copy_(x)
            s["list"] = np.zeros(CAP, dtype=_lib.CAND_DTYPE)
            _lib.af_search_reserve(p.handle, c["nsamp"], CAP)
            return s
        s["x"] = x
        s["plane"] = torch.empty((c["ndm"], nout), dtype=torch.int32, device=dev)
        s["stats"] = torch.empty((c["ndm"], 2), dtype=torch.int64, device=dev)
        p.reserve(c["nsamp"])
        if k == "search":
            s["snr"] = torch.empty((c["ndm"], nout), dtype=torch.float32, device=dev)
            s["bw"] = torch.empty((c["ndm"], nout), dtype=torch.uint8, device=dev)
            s["list"] = np.zeros(CAP, dtype=_lib.CAND_DTYPE)
            s["cands"] = torch.empty((CAP, _lib.CAND_DTYPE.itemsize), dtype=torch.uint8, device=dev)
            s["count"] = torch.empty(1, dtype=torch.int32, device=dev)
        if k == "classify":
            p.dedisperse(x, plane=s["plane"])
            a = _candidates(c, nout, seed)
            s["list"] = torch.from_numpy(a.view(np.uint8).reshape(c["n"], a.itemsize)).to(dev)
            s["cut"] = torch.empty((c["n"], 64, 64, 2), dtype=torch.bfloat16, device=dev)
            s["logits"] = torch.empty((c["n"], 2), device=dev)
            s["prob"] = torch.empty(c["n"], device=dev)
            s["model"] = _model(c["n"], _trained())
    elif k == "stream":
        dms = _dms(c)
        h = _lib.af_stream_open(2, c["nchan"], F_LO, F_HI, c["tsamp_us"] * 1e-6, dms, c["nsamp"], _widths(c), 8.0,
                                CAP, hbm_budget=24 << 30, max_slots=2)
        s["engine"] = _Handle(h, _lib.af_stream_close)
        s["model"] = _model(256, _trained())
        s["list"] = [dict(cands=np.zeros(CAP, dtype=_lib.CAND_DTYPE), reps=np.zeros(256, dtype=_lib.CAND_DTYPE),
                          prob=np.zeros(256, dtype=np.float32)) for _ in range(2)]
        hop, dmax, _ = _lib.af_stream_info(h)
        s["hop"], s["seq"], s["chunk"] = hop, 0, []
        # each beam's stream repeats one hop of samples, so that every window holds the same data (dmax < hop)
        for b in range(2):
            x = _filterbank(c, 2 * seed + b, hop=hop)
            a = torch.empty((c["nchan"], hop), dtype=torch.uint8, pin_memory=True)
            a.copy_(x)
            first = torch.cat([x[:, hop - dmax:], x], dim=1).cpu().numpy()
            _lib.af_stream_push(h, b, first, 0)
            _lib.af_stream_release(h, _lib.af_stream_poll(h)["slot"])
            s["chunk"].append(a)
    elif k == "prep":
        c["tsamp_us"], c["ndm"], c["dm_step"] = 49.152, 2, 100.0
        s["x"] = synth.filterbank_torch(c["nchan"], c["nsamp"], seed,
                                        rfi=synth.RFI(narrow_channels=(3, c["nchan"] // 2),
                                                      bursts=((c["nsamp"] // 3, 20, 40.0),)))
        s["z"] = torch.empty_like(s["x"])
        s["low"] = torch.empty((c["nchan"], -(-c["nsamp"] // c["factor"])), dtype=torch.uint8, device=dev)
    elif k in ("robust", "grid"):
        s["plane"] = _plane(c, seed)
        if k == "robust":
            # any plan with these rows and channels serves the row statistics and the boxcar
            s["plan"] = Plan(c["nchan"], F_LO, F_HI, 49.152e-6, np.arange(c["ndm"]) * 1.0)
            s["stats"] = torch.empty((c["ndm"], 2), dtype=torch.int64, device=dev)
            s["snr"] = torch.empty((c["ndm"], c["nout"]), dtype=torch.float32, device=dev)
            s["bw"] = torch.empty((c["ndm"], c["nout"]), dtype=torch.uint8, device=dev)
        else:
            n = -(-c["nout"] // c["ns"])
            s["img"] = torch.empty((n, c["m"], c["m"]), dtype=torch.uint8, device=dev)
            s["work"] = torch.empty((n, 2), dtype=torch.int64, device=dev)
    elif k == "infer":
        s["model"] = _model(c["n"], _trained())
        s["x"], _ = _images(c["n"], seed)
        s["logits"] = torch.empty((c["n"], 2), device=dev)
        s["prob"] = torch.empty(c["n"], device=dev)
    else:
        s["model"] = _model(c["n"], _initial(seed))
        s["x"], s["y"] = _images(c["n"] * c["steps"], seed)
        s["loss"] = torch.empty(c["steps"], device=dev)
    return s


# ---- one pass ---------------------------------------------------------------

def _fields(a):
    return {k: a[k] for k in ("dm_idx", "t", "width", "snr")}


def _into(buf, found):
    """The program's own list, of a length that does not depend on what was found (zeros behind it)."""
    buf[:len(found)] = found
    buf[len(found):] = 0
    return _fields(buf)


def run(s):
    k = s["kind"]
    stream = torch.cuda.current_stream().cuda_stream
    if k == "search":
        p, w = s["plan"], _widths(s)
        p.dedisperse(s["x"], plane=s["plane"], stats=s["stats"])
        p.boxcar_snr(s["plane"], w, stats=s["stats"], snr=s["snr"], bw=s["bw"])
        p.candidates(s["snr"], s["bw"], w, 8.0, cap=CAP, out=s["cands"], count=s["count"])
        found, total = Plan.cands_to_numpy(s["cands"], s["count"])
        return dict(plane=s["plane"], stats=s["stats"], snr=s["snr"], bw=s["bw"], total=total,
                    cands=_into(s["list"], found))
    if k == "host":
        _, total = _lib.af_search(s["plan"].handle, s["h"].data_ptr(), s["nsamp"], _widths(s), 8.0, CAP,
                                  stream=stream, out=s["list"])
        return dict(total=total, cands=_fields(s["list"]))
    if k == "stream":
        h, out = s["engine"].h, {}
        s["seq"] += 1
        for b in range(2):
            _lib.af_stream_push(h, b, (s["chunk"][b].data_ptr(), s["hop"], s["hop"]), s["seq"])
        for _ in range(2):
            r = _lib.af_stream_poll(h)
            reps = _lib.af_stream_cluster(h, r["cands"])
            prob = _lib.af_stream_classify(h, r["slot"], s["model"].h, reps)
            _lib.af_stream_release(h, r["slot"])
            own = s["list"][r["beam"]]
            own["prob"][:] = 0.0
            own["prob"][:len(prob)] = prob
            out["beam%d" % r["beam"]] = dict(total=r["total"], cands=_into(own["cands"], r["cands"]),
                                             reps=_into(own["reps"], reps), prob=own["prob"])
        return out
    if k == "subband":
        s["plan"].dedisperse(s["x"], plane=s["plane"], stats=s["stats"])
        return dict(plane=s["plane"], stats=s["stats"])
    if k == "prep":
        _lib.af_zerodm(s["x"].data_ptr(), s["nchan"], s["nsamp"], s["z"].data_ptr(), stream)
        _lib.af_downsample(s["z"].data_ptr(), s["nchan"], s["nsamp"], s["factor"], s["low"].data_ptr(), stream)
        return dict(filtered=s["z"], low=s["low"])
    if k == "robust":
        h, y, w = s["plan"].handle, s["plane"], _widths(s)
        _lib.af_rowstats_robust(h, y.data_ptr(), s["nout"], s["stats"].data_ptr(), stream)
        _lib.af_boxcar_snr_robust(h, y.data_ptr(), s["nout"], s["stats"].data_ptr(), w, s["snr"].data_ptr(),
                                  s["bw"].data_ptr(), stream)
        return dict(stats=s["stats"], snr=s["snr"], bw=s["bw"])
    if k == "grid":
        _lib.af_grid(s["plane"].data_ptr(), s["ndm"], s["nout"], s["ns"], s["m"], s["img"].data_ptr(),
                     s["work"].data_ptr(), stream)
        return s["img"]
    if k == "classify":
        _lib.af_cutouts(s["plan"].handle, s["x"].data_ptr(), s["nsamp"], s["plane"].data_ptr(), s["nout"],
                        s["list"].data_ptr(), s["n"], s["cut"].data_ptr(), stream)
        _lib.af_model_forward(s["model"].h, s["cut"].data_ptr(), s["n"], s["logits"].data_ptr(),
                              s["prob"].data_ptr(), stream)
        return dict(cut=s["cut"], logits=s["logits"], prob=s["prob"])
    if k == "infer":
        _lib.af_model_forward(s["model"].h, s["x"].data_ptr(), s["n"], s["logits"].data_ptr(), s["prob"].data_ptr(),
                              stream)
        return dict(logits=s["logits"], prob=s["prob"])
    n, m = s["n"], s["model"].h
    for i in range(s["steps"]):
        _lib.af_train_step(m, s["x"][i * n:].data_ptr(), s["y"][i * n:].data_ptr(), n, 1e-4, s["loss"][i:].data_ptr(),
                           stream)
    # what the training loop reads at the end of an epoch (grads: the last batch's)
    return dict(loss=s["loss"], grads=_lib.af_model_get_grads(m), params=_lib.af_model_get_params(m))


def work(case):
    c = case
    k = c["kind"]
    if k in ("search", "host", "stream", "subband"):
        dmax = int(_delays(c).max())
        nout, beams = c["nsamp"] - dmax, 2 if k == "stream" else 1
        read = c["nchan"] * (nout if k == "stream" else c["nsamp"])
        write = {"search": 9 * c["ndm"] * nout, "subband": 4 * c["ndm"] * nout}.get(k, 0)
        # a host search's result is its candidate list; the sum over channels is counted as defined, one addition each
        adds = c["ndm"] * c["nchan"] * nout if k != "subband" else \
            -(-c["ndm"] // c["n0"]) * c["nchan"] * nout + c["ndm"] * c["nsub"] * nout
        return dict(bytes=beams * (read + write), flops=beams * adds)
    if k == "prep":
        n = c["nchan"] * c["nsamp"]
        return dict(bytes=2 * n + n / c["factor"], flops=2 * n)
    if k == "robust":
        n = c["ndm"] * c["nout"]
        return dict(bytes=9 * n, flops=3 * n * len(_widths(c)))
    if k == "grid":
        n = c["ndm"] * c["nout"]
        return dict(bytes=4 * n + c["m"] ** 2 * -(-c["nout"] // c["ns"]), flops=2 * n)
    images = c["n"] * c.get("steps", 1)
    flops = sum(2 * (64 >> l) ** 2 * 9 * CH[l] * CH[l + 1] for l in range(3)) * images
    if k == "classify":
        # mean over the drawn widths 1..256 of the samples in a cut-out's windows
        span = 64 * sum(max(1, (1 << e) // 2) for e in range(9)) / 9
        return dict(bytes=c["n"] * (span * (4 * 64 + c["nchan"]) + 64 * 64 * 4), flops=flops)
    return dict(bytes=images * 64 * 64 * 4, flops=flops * (3 if k == "train" else 1))


# ---- the same in 64 bits -------------------------------------------------------

def _exact_plane(x, D, nout):
    """Y[d][t] = sum_c x[c][t + D[d][c]], channel by channel, in exact integers."""
    D = torch.from_numpy(D).to(x.device)
    y = torch.zeros((D.shape[0], nout), dtype=torch.int32, device=x.device)
    for ch in range(x.shape[0]):
        y += x[ch].unfold(0, nout, 1)[D[:, ch]]
    return y


def _exact_snr(y, widths, loc, scale):
    """Best over widths of (window sum - w loc) / (scale sqrt(w)), row by row, float64."""
    out = torch.full(y.shape, -math.inf, dtype=torch.float64, device=y.device)
    n = y.shape[1]
    for d in range(y.shape[0]):
        P = torch.nn.functional.pad(torch.cumsum(y[d].long(), 0), (1, 0))
        for w in widths:
            if w > n:
                break
            B = (P[w:] - P[:-w]).double()
            v = (B - w * loc[d]) / (scale[d] * math.sqrt(w)) if float(scale[d]) > 0 else torch.zeros_like(B)
            out[d, :n - w + 1] = torch.maximum(out[d, :n - w + 1], v)
    return out


def _network(p, x):
    h = x.permute(0, 3, 1, 2)
    for l in range(3):
        h = torch.nn.functional.conv2d(h, p["w%d" % l].permute(0, 3, 1, 2), p["b%d" % l], padding=1)
        h = torch.nn.functional.max_pool2d(torch.relu(h), 2)
    return h.mean(dim=(2, 3)) @ p["fw"].T + p["fb"]


def _split(flat, grad=False):
    p, o = {}, 0
    for name, shape in SIZES:
        k = int(np.prod(shape))
        p[name] = torch.from_numpy(flat[o:o + k].astype(np.float64)).cuda().reshape(shape).requires_grad_(grad)
        o += k
    return p


def _exact_cutouts(c, x, y, D, cands):
    out = torch.zeros((len(cands), 64, 64, 2), dtype=torch.float64, device=x.device)
    nout = y.shape[1]
    g = c["nchan"] // 64
    D = torch.from_numpy(D).to(x.device)
    rows = torch.arange(c["nchan"], device=x.device)[:, None]
    for i, a in enumerate(cands):
        d, t, b = int(a["dm_idx"]), int(a["t"]), max(1, int(a["width"]) // 2)
        s = torch.arange(t - 32 * b, t + 32 * b, device=x.device)
        s0, ok = s.clamp(0, nout - 1), (s >= 0) & (s < nout)
        lo, hi = max(0, d - 32), min(c["ndm"], d + 32)
        u = torch.zeros((64, 64), dtype=torch.int64, device=x.device)
        u[lo - d + 32:hi - d + 32] = (y[lo:hi][:, s0] * ok).long().reshape(hi - lo, 64, b).sum(2)
        v = (x[rows, s0[None, :] + D[d][:, None]] * ok).reshape(64, g, 64, b).sum((1, 3))
        for k, z in enumerate((u, v)):
            z = z.double()
            out[i, :, :, k] = (z - z.min()) / (z.max() - z.min() + 1e-6)
    return out


def exact(case, seed):
    c = dict(case)
    k = c["kind"]
    if k in ("search", "classify"):
        D = _delays(c)
        nout = c["nsamp"] - int(D.max())
        if k == "classify" and c["ndm"] * c["nchan"] * nout > 2e11:
            return None
        x = _filterbank(c, seed)
        y = _exact_plane(x, D, nout)
        if k == "search":
            loc = y.double().mean(1)
            scale = (y.double() - loc[:, None]).square().mean(1).sqrt() if y.numel() < 1 << 24 else \
                torch.stack([(r.double() - m).square().mean().sqrt() for r, m in zip(y, loc)])
            return dict(plane=None, stats=None, snr=_exact_snr(y, _widths(c), loc, scale), bw=None, total=None,
                        cands=None)
        cut = _exact_cutouts(c, x, y, D, _candidates(c, nout, seed))
        z = _network(_split(_trained()), cut)
        return dict(cut=cut, logits=z, prob=torch.softmax(z, 1)[:, 1])
    if k == "robust":
        y = _plane(c, seed)
        mid = (c["nout"] - 1) // 2
        med = torch.stack([r.sort().values[mid] for r in y])
        mad = torch.stack([(r - m).abs().sort().values[mid] for r, m in zip(y, med)])
        return dict(stats=None, bw=None,
                    snr=_exact_snr(y, _widths(c), med.double(), 1.482602218505602 * mad.double()))
    if k == "infer":
        x, _ = _images(c["n"], seed)
        z = torch.cat([_network(_split(_trained()), b.double()) for b in x.split(512)])
        return dict(logits=z, prob=torch.softmax(z, 1)[:, 1])
    if k == "train":
        n, lr = c["n"], 1e-4
        x, y = _images(n * c["steps"], seed)
        p = _split(_initial(seed), grad=True)
        names = [name for name, _ in SIZES]
        m, v = ({a: torch.zeros_like(p[a]) for a in names} for _ in range(2))
        loss = []
        for i in range(c["steps"]):
            grads, tot = {a: torch.zeros_like(p[a]) for a in names}, 0.0
            for xb, yb in zip(x[i * n:(i + 1) * n].split(512), y[i * n:(i + 1) * n].split(512)):
                one = torch.nn.functional.cross_entropy(_network(p, xb.double()), yb.long(), reduction="sum") / n
                for a, g in zip(names, torch.autograd.grad(one, [p[a] for a in names])):
                    grads[a] += g
                tot += one.detach()
            loss.append(tot)
            with torch.no_grad():
                for a in names:
                    m[a].mul_(0.9).add_(grads[a], alpha=0.1)
                    v[a].mul_(0.999).add_(grads[a].square(), alpha=0.001)
                    hat = (v[a] / (1 - 0.999 ** (i + 1))).sqrt() + 1e-8
                    p[a].sub_(lr / (1 - 0.9 ** (i + 1)) * m[a] / hat)
        flat = [torch.cat([q[a].detach().reshape(-1) for a in names]).cpu().numpy() for q in (grads, p)]
        return dict(loss=torch.stack(loss), grads=flat[0], params=flat[1])
    return None
