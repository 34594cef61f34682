"""The work that users of this library have it do, as cases that can be timed and compared.

A case is a dict of plain values.  `prepare` draws its inputs from a seed and makes what a calling program keeps
(catalogs, grid, page-locked result arrays, a recorded batch, a vetter with its weights), `run` makes one pass
through the public entry points of `paper_2509_26279_gb300.sas`, `work` says what such a pass cannot do without, and
`exact` gives the networks' results in 64 bits.

The kinds of case:
  search       sas_stack (or its weighted form) on one field, candidates and ids copied to the caller's arrays
  batch        one replay of a recorded batch of uneven fields, every field vetted, the lists copied out
  tracks       cluster finding on a finished search, then refinement and gathering of its clusters
  vet_field    ownership selection, stamps and scores of one finished search
  vet_forward  scores of stamps that are on the device already
  vet_grad     loss and gradients of one training batch
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2509_26279_gb300 import sas, vetting
from paper_2509_26279_gb300 import workloads as W

MAX_CANDIDATES, MAX_IDS = 1 << 18, 3 << 20  # the caller's result arrays (page-locked where a search fills them)
MAX_SCORED = 1 << 17                        # items of a vetted batch
MAX_KEPT = 1 << 13                          # stamps of one vetted field
MAX_TRACKS = 1000                           # clusters, the library's own cut


def _field_case(name, width, height, epochs, span_h, noise, movers, speeds, p, nvx, nvy, step, bin_mpx, n_min, **more):
    c = dict(name=name, kind="search", width=width, height=height, epochs=epochs, span_h=span_h, noise=noise,
             movers=movers, speed_lo=speeds[0], speed_hi=speeds[1], p_hi=p[0], p_lo=p[1], nvx=nvx, nvy=nvy, step=step,
             bin_mpx=bin_mpx, n_min=n_min)
    c.update(more)
    return c


def _tno(name, **more):
    """The DECam TNO field: 2048 x 4096 px, 100 epochs in 4 h, 111 x 111 velocities."""
    return _field_case(name, 2048, 4096, 100, 4.0, 3000, 200, (0.5, 20.0), (0.9, 0.3), 111, 111, 364, 2000, 25, **more)


def listed():
    return [
        # The smallest search: a cut-out of 512 px held in host arrays; launches and latency are all there is.
        _field_case("search_tiny", 512, 512, 20, 4.0, 200, 3, (1.0, 10.0), (0.6, 0.6), 21, 21, 1000, 4000, 8, host=True),
        # The ordinary search of one CCD, catalog on the device.
        _tno("search_tno"),
        # A chip of odd size from host arrays: odd epochs, an odd bin, a lattice that is not square and only its
        # annulus of rates searched.
        _field_case("search_ragged", 1531, 2777, 47, 3.3, 1733, 77, (1.0, 15.0), (0.85, 0.4), 83, 61, 457, 2501, 13,
                    speed_min=900, speed_max=16100, host=True),
        # The largest search: a million velocities up to 300 px/h over a dense field.
        _field_case("search_fast", 2048, 4096, 60, 1.5, 5000, 100, (20.0, 300.0), (0.9, 0.3), 1001, 1001, 600, 3000, 15),
        # A search for fainter movers beside the complete list at n_min: peaks of the super-bins at a lower threshold.
        _field_case("search_low", 2048, 4096, 120, 4.0, 2400, 200, (0.5, 20.0), (0.9, 0.3), 111, 111, 364, 2000, 30, n_low=20),
        # Likelihood-weighted stacking of the TNO field.
        _tno("search_weighted", weighted=True, s_min=1000),
        # A night's uneven CCDs in one recorded pass, peaks alone at a lowered threshold, every candidate scored.
        dict(name="batch_vet", kind="batch", fields=12, shapes=4, noise_lo=1000, noise_hi=8000, half=55, step=364),
        # From a finished TNO search to refined trajectories.
        _tno("tracks_tno", kind="tracks"),
        # Scoring what one search at a low threshold found.
        _field_case("vet_field", 2048, 4096, 90, 4.0, 2900, 200, (0.5, 20.0), (0.9, 0.06), 111, 111, 364, 2000, 9, kind="vet_field"),
        # Scoring a large pool of stamps.
        dict(name="vet_forward", kind="vet_forward", n=32768, max_batch=32768),
        # One training batch of the size that vetting.train takes, gathered from a pool through an index.
        dict(name="vet_grad", kind="vet_grad", n=512, max_batch=512, pool=20000),
        # A large training batch.
        dict(name="vet_grad_large", kind="vet_grad", n=4096, max_batch=4096, pool=0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _noise_n_min(n, bins, velocities, budget):
    """The smallest threshold that uniform noise passes in fewer than `budget` cells."""
    lam = n / bins
    k, term = 0, math.exp(-lam)
    sf = 1.0
    while sf * bins * velocities > budget:
        sf -= term
        k += 1
        term *= lam / k
        if sf < 1e-12:
            sf = term
    return max(k, 3)


def _draw_field(rng, kind):
    while True:
        epochs = rng.randint(11, 150)
        span = round(rng.uniform(1.0, 6.0), 2)
        width, height = int(_log(rng, 400, 2300)), int(_log(rng, 400, 4400))
        noise = max(40, int(_log(rng, 1.2e-4, 9.5e-4) * width * height))
        bin_mpx = int(_log(rng, 1600, 4200))
        step = max(100, int(rng.uniform(0.3, 1.0) * bin_mpx / span))
        nvx, nvy = int(_log(rng, 9, 500)), int(_log(rng, 9, 500))
        n = noise * epochs
        if kind != "search" and nvx * nvy > 14000:
            continue
        if n * nvx * nvy > 8e10:
            continue
        bins = width * height * 1e6 / bin_mpx ** 2
        n_min = max(_noise_n_min(n, bins, nvx * nvy, 1000), -(-epochs // 4), 4)
        if n_min > 0.8 * epochs:
            continue
        top = min(nvx, nvy) // 2 * step / 1000
        movers = rng.randint(2, int(200 * min(1.0, (step * span / bin_mpx / 0.6) ** 2)))
        c = _field_case("", width, height, epochs, span, noise, movers, (0.05 * top, top), (0.9, 0.3), nvx, nvy, step, bin_mpx,
                        n_min, kind=kind)
        del c["name"]
        return c


def draw(rng):
    kind = rng.choice(["search", "search", "search", "low", "weighted", "batch", "tracks", "vet_field", "vet_forward",
                       "vet_forward", "vet_grad", "vet_grad"])
    if kind == "vet_forward":
        n = int(_log(rng, 33, 32768))
        return dict(kind=kind, n=n, max_batch=rng.choice([1024, 4096, 32768]))
    if kind == "vet_grad":
        n = int(_log(rng, 17, 4096))
        return dict(kind=kind, n=n, max_batch=n, pool=rng.choice([0, 2 * n + 1]))
    if kind == "batch":
        return dict(kind=kind, fields=rng.randint(3, 14), shapes=rng.randint(10, 1 << 20), noise_lo=700,
                    noise_hi=int(_log(rng, 2000, 8000)), half=rng.randint(20, 60), step=rng.randint(300, 500))
    if kind in ("tracks", "vet_field"):
        return _draw_field(rng, kind)
    c = _draw_field(rng, "search")
    c["host"] = rng.random() < 0.4
    if kind == "low":
        bins = c["width"] * c["height"] * 1e6 / c["bin_mpx"] ** 2
        floor = _noise_n_min(c["noise"] * c["epochs"], bins, c["nvx"] * c["nvy"], 10000)
        c["n_low"] = min(c["n_min"], max(floor, c["n_min"] - rng.randint(1, 10)))
        c["peaks_only"] = rng.random() < 0.5
    elif kind == "weighted":
        c["weighted"], c["s_min"] = True, 42 * c["n_min"]
    elif rng.random() < 0.3:
        top = max(c["nvx"], c["nvy"]) // 2 * c["step"]
        c["speed_min"], c["speed_max"] = int(0.05 * top), int(0.95 * top)
    return c


def _recipe(case):
    return W.FieldRecipe(case["width"], case["height"], case["epochs"], case["span_h"], case["noise"], case["movers"],
                         (case["speed_lo"], case["speed_hi"]), (case["p_hi"], case["p_lo"]))


def _grid(case):
    nvx, nvy, step, b = case["nvx"], case["nvy"], case["step"], case["bin_mpx"]
    return sas.Grid(vx0=-(nvx // 2) * step, vy0=-(nvy // 2) * step, dvx=step, dvy=step, nvx=nvx, nvy=nvy, x_min=0, y_min=0,
                    nbx=-(-case["width"] * 1000 // b), nby=-(-case["height"] * 1000 // b), bin=b,
                    speed_min=case.get("speed_min", 0), speed_max=case.get("speed_max", 0))


def _device(a):
    return torch.from_numpy(a.view(np.int16) if a.dtype == np.uint16 else a).cuda()


def _vetter(seed, max_batch):
    v = sas.Vetter(0, max_batch)
    v.set_state(_params(seed))
    return v


def _params(seed):
    """He-normal weights and small biases: what training starts from and stays near."""
    p = vetting.init_params(seed)
    rng = np.random.default_rng([seed, 1])
    at = 0
    for name, shape in vetting.PARAMS:
        k = int(np.prod(shape))
        if name.endswith(".b"):
            p[at:at + k] = rng.normal(0.0, 0.02, k)
        at += k
    return p


def _stamps(n, seed):
    """Count stamps as searches give them: noise counts of one background per stamp, and in every second one a mover,
    a peak at the centre that fades over the neighbouring velocities.  Labels 1 for movers."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    uni = lambda *s: torch.rand(s, generator=g, device="cuda")  # noqa: E731
    label = (uni(n) < 0.5).float()
    out = torch.empty((n, 9, 15, 15), dtype=torch.int16, device="cuda")
    at = torch.arange(15, device="cuda", dtype=torch.float32) - 7
    q = torch.arange(9, device="cuda")
    dy, dx = (q // 3 - 1).float(), (q % 3 - 1).float()
    for a in range(0, n, 4096):
        b = min(n, a + 4096)
        m = b - a
        back = 0.03 * 20 ** uni(m)
        height = label[a:b] * (4 + 60 * uni(m)) + (1 - label[a:b]) * 6 * uni(m)
        cx, cy = uni(m) - 0.5, uni(m) - 0.5
        wide = 0.5 + 0.4 * uni(m)
        sx = (at[None, None, :] - cx[:, None, None] - 0.7 * dx[None, :, None]) / wide[:, None, None]
        sy = (at[None, None, :] - cy[:, None, None] - 0.7 * dy[None, :, None]) / wide[:, None, None]
        fade = 0.75 ** (dx.abs() + dy.abs())
        mean = back[:, None, None, None] + height[:, None, None, None] * fade[None, :, None, None] * \
            torch.exp(-0.5 * sx ** 2)[:, :, None, :] * torch.exp(-0.5 * sy ** 2)[:, :, :, None]
        out[a:b] = torch.poisson(mean, generator=g).to(torch.int16)
    return out, label


def _pool_index(case, seed):
    """The batch's stamps within the pool (a shuffled mini-batch), or None for the first n."""
    if not case["pool"]:
        return None
    return np.random.default_rng([seed, 2]).permutation(case["pool"])[:case["n"]].astype(np.int32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "vet_forward":
        stamps, _ = _stamps(case["n"], seed)
        return dict(case=case, stamps=stamps, vetter=_vetter(seed, case["max_batch"]),
                    logits=torch.zeros(case["n"], device="cuda"))
    if kind == "vet_grad":
        stamps, labels = _stamps(case["pool"] or case["n"], seed)
        idx = _pool_index(case, seed)
        return dict(case=case, stamps=stamps, labels=labels, index=None if idx is None else torch.from_numpy(idx).cuda(),
                    vetter=_vetter(seed, case["max_batch"]), grad=torch.zeros(sas.vet_num_params(), device="cuda"),
                    loss=torch.zeros(1, device="cuda"))
    if kind == "batch":
        return _prepare_batch(case, seed)
    cat = W.make_catalog(_recipe(case), seed)
    s = dict(case=case, grid=_grid(case), cat=cat)
    if case.get("host"):
        s["x"], s["y"], s["e"] = cat.x, cat.y, cat.epoch
    else:
        s["x"], s["y"], s["e"] = _device(cat.x), _device(cat.y), _device(cat.epoch)
    if case.get("weighted"):
        w = W.snr_weights(cat, seed=seed)
        s["w"] = w if case.get("host") else torch.from_numpy(w).cuda()
    s["opts"] = sas.make_opts(n_low=case["n_low"], peaks_only=case.get("peaks_only", 0)) if case.get("n_low") else None
    if kind == "search":
        s["cands"], s["ids"] = _host_lists(MAX_CANDIDATES, MAX_IDS)
    else:
        s["res"] = _search(s)
        if kind == "vet_field":
            s["vetter"] = _vetter(seed, 4096)
            s["idx"] = torch.zeros(MAX_CANDIDATES, dtype=torch.int32, device="cuda")
            s["stamps"] = torch.zeros((MAX_KEPT, 9, 15, 15), dtype=torch.int16, device="cuda")
            s["logits"] = torch.zeros(MAX_KEPT, device="cuda")
        else:
            s["cands"], s["ids"] = _host_lists(MAX_TRACKS, MAX_IDS // 16)
            s["tracks"], s["track_ids"] = np.zeros(MAX_TRACKS, sas.TRACK_DTYPE), np.zeros(MAX_IDS // 16, np.int32)
    return s


def _host_lists(candidates, ids):
    """Page-locked arrays for a search's candidates and ids, reused from pass to pass."""
    size = lambda n: torch.zeros(n, dtype=torch.uint8, pin_memory=True).numpy()  # noqa: E731
    return size(candidates * 32).view(sas.CANDIDATE_DTYPE), size(ids * 4).view(np.uint32)


def _batch_shapes(case):
    """Epochs and noise of each field, the same for every seed."""
    rng = np.random.default_rng(case["shapes"])
    return [(int(rng.integers(20, 151)), int(round(math.exp(rng.uniform(math.log(case["noise_lo"]), math.log(case["noise_hi"]))))))
            for _ in range(case["fields"])]


def _prepare_batch(case, seed):
    fields, opts, cats = [], [], []
    for f, (epochs, noise) in enumerate(_batch_shapes(case)):
        cat = W.make_catalog(W.FieldRecipe(2048, 4096, epochs, 4.0, noise, 200, (0.5, 20.0), (0.9, 0.3)), seed * 1000 + f)
        spec = W.field_grid(2048, 4096, 2000, case["step"], case["half"])
        n_min = -(-epochs // 4)
        fields.append((sas.Grid(spec), _device(cat.x), _device(cat.y), _device(cat.epoch), cat.t, cat.ticks_per_hour, n_min))
        opts.append(sas.make_opts(n_low=vetting.lowered_threshold(epochs, n_min, cat.n, spec), peaks_only=1))
        cats.append(cat)
    new = lambda dtype: torch.zeros(MAX_SCORED, dtype=dtype, device="cuda")  # noqa: E731
    return dict(case=case, fields=fields, cats=cats, batch=sas.Batch(fields, opts), vetter=_vetter(seed, 4096),
                field=new(torch.int32), cand=new(torch.int32), logit=new(torch.float32),
                cands=np.zeros(MAX_CANDIDATES, sas.CANDIDATE_DTYPE), ids=np.zeros(MAX_IDS, np.uint32))


def _search(s):
    c, cat = s["case"], s["cat"]
    on_device = not c.get("host")
    if c.get("weighted"):
        return sas.sas_stack_weighted(s["grid"], s["x"], s["y"], s["e"], s["w"], cat.t, cat.ticks_per_hour, c["s_min"],
                                      on_device=on_device)
    return sas.sas_stack(s["grid"], s["x"], s["y"], s["e"], cat.t, cat.ticks_per_hour, c["n_min"], on_device=on_device,
                         opts=s["opts"])


def _plain(records):
    """Candidate records as whole numbers, eight to a record."""
    return records.view(np.int32).reshape(-1, 8)


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "search":
        res = _search(s)
        cands, ids = res.candidates(out=(s["cands"], s["ids"]))
        pairs = res.info()["n_pairs"]
        res.free()
        return dict(candidates=_plain(s["cands"]), ids=s["ids"].view(np.int32), sizes=[len(cands), len(ids), pairs])
    if kind == "batch":
        b = s["batch"]
        b.run()
        k = b.vet(s["vetter"], s["field"], s["cand"], s["logit"], MAX_SCORED)
        ends, nc, ni = [], 0, 0
        for f in range(b.n_fields):  # the night's lists, one behind the other
            cands, ids = b.candidates(f)
            s["cands"][nc:nc + len(cands)] = cands
            s["ids"][ni:ni + len(ids)] = ids
            nc, ni = nc + len(cands), ni + len(ids)
            ends.append((nc, ni))
        return dict(candidates=_plain(s["cands"]), ids=s["ids"].view(np.int32), ends=np.array(ends), scored=k, field=s["field"],
                    candidate=s["cand"], logit=s["logit"])
    if kind == "tracks":
        clusters = sas.sas_peel(s["res"], c["n_min"])
        found = sas.sas_refine(s["res"], clusters, seed=1)
        cands, ids = clusters.candidates(out=(s["cands"], s["ids"]))
        tr, tids = found.tracks()
        found.free()
        clusters.free()
        s["tracks"][:len(tr)], s["track_ids"][:len(tids)] = tr, tids.view(np.int32)
        tr = s["tracks"]
        return dict(clusters=_plain(s["cands"]), ids=s["ids"].view(np.int32), track_ids=s["track_ids"],
                    sizes=[len(cands), len(ids), len(tids)],
                    line=np.stack([tr[k] for k in ("vx", "vy", "x0", "y0")]),
                    spread=np.stack([tr[k] for k in ("res_xx", "res_xy", "res_yy")]), det=tr["det"],
                    state=np.stack([tr[k].astype(np.int32) for k in ("status", "iterations", "h", "n_points", "id_len", "cluster")]))
    if kind == "vet_field":
        kept = sas.sas_owned(s["res"], s["idx"], c["n_min"])
        k = min(kept, MAX_KEPT)
        sas.sas_stamps_indexed(s["res"], s["idx"], k, s["stamps"])
        s["vetter"].forward(s["stamps"], k, s["logits"])
        return dict(kept=kept, idx=s["idx"], stamps=s["stamps"], logits=s["logits"])
    if kind == "vet_forward":
        s["vetter"].forward(s["stamps"], c["n"], s["logits"])
        return dict(logits=s["logits"])
    s["vetter"].gradients(s["stamps"], s["labels"], c["n"], s["grad"], s["loss"], index=s["index"])
    return dict(grad=_layers(s["grad"]), loss=s["loss"])


def _layers(flat):
    """The flat gradient's parameter tensors."""
    out, at = {}, 0
    for name, shape in vetting.PARAMS:
        k = int(np.prod(shape))
        out[name] = flat[at:at + k]
        at += k
    return out


# multiply-adds of one stamp: conv1, conv2, conv3, fc1, fc2
_MACS = (13 * 13 * 32 * 81, 11 * 11 * 32 * 288, 9 * 9 * 32 * 288, 2592 * 64, 64)


def _search_work(epochs, noise, movers, velocities, weighted):
    """The catalog once and a record and ids of each mover; one addition for each detection and velocity (integers)."""
    n = epochs * (noise + 0.5 * movers)
    return dict(bytes=n * (11 if weighted else 10) + movers * (32 + 4 * epochs / 2), flops=n * velocities)


def work(case):
    kind = case["kind"]
    if kind == "search":
        return _search_work(case["epochs"], case["noise"], case["movers"], case["nvx"] * case["nvy"], case.get("weighted"))
    if kind == "batch":
        v = (2 * case["half"] + 1) ** 2
        each = [_search_work(e, n, 200, v, False) for e, n in _batch_shapes(case)]
        return dict(bytes=sum(w["bytes"] for w in each), flops=sum(w["flops"] for w in each))
    if kind == "tracks":
        # per mover: two fits of 500 starts with two C-steps each, over half the epochs' points, about 30 operations a point
        points = case["epochs"] / 2
        return dict(bytes=case["movers"] * points * 40 + 10.0 * case["epochs"] * case["noise"],
                    flops=case["movers"] * 2 * 500 * 2 * points * 30)
    n = case["n"] if kind != "vet_field" else 2 * case["movers"]
    flops = 2.0 * n * sum(_MACS)
    size = n * 2025 * 2 + n * 4 + 4 * sas.vet_num_params()
    if kind == "vet_grad":  # the backward: weight gradients of all layers, input gradients of all but the first
        flops += 2.0 * n * (2 * sum(_MACS) - _MACS[0])
        size += 4 * sas.vet_num_params()
    return dict(bytes=size, flops=flops)


def _bf16(x):
    """x as the library stores it (BF16), straight through for gradients."""
    return x + (x.detach().to(torch.bfloat16).to(x.dtype) - x.detach())


def _logits64(p, stamps):
    """The network of include/sas.h in 64 bits, with the BF16 storage of weights and activations that it states."""
    n = stamps.shape[0]
    a = _bf16(stamps.to(torch.float64) / 16)
    w = {k: _bf16(v) for k, v in p.items()}
    for layer, ci, h in (("conv1", 9, 13), ("conv2", 32, 11), ("conv3", 32, 9)):
        cols = F.unfold(a, 3)
        a = torch.matmul(w[layer + ".w"].reshape(32, ci * 9), cols) + w[layer + ".b"][None, :, None]
        a = _bf16(torch.relu(a)).reshape(n, 32, h, h)
    a = _bf16(torch.relu(a.reshape(n, -1) @ w["fc1.w"].reshape(64, 2592).T + w["fc1.b"]))
    return a @ w["fc2.w"] + w["fc2.b"]


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("vet_forward", "vet_grad"):
        return None  # whole numbers, and scores of stamps that the search cuts; and the robust fits of "tracks", which plain numpy takes minutes for
    p, at = {}, 0
    flat = torch.from_numpy(_params(seed)).cuda().double()
    for name, shape in vetting.PARAMS:
        k = int(np.prod(shape))
        p[name] = flat[at:at + k].reshape(shape).clone().requires_grad_(kind == "vet_grad")
        at += k
    stamps, labels = _stamps(case.get("pool") or case["n"], seed)
    if kind == "vet_forward":
        with torch.no_grad():
            return dict(logits=torch.cat([_logits64(p, stamps[a:a + 2048]) for a in range(0, case["n"], 2048)]))
    idx = _pool_index(case, seed)
    if idx is not None:
        at = torch.from_numpy(idx).long().cuda()
        stamps, labels = stamps[at], labels[at]
    n, total = case["n"], 0.0
    for a in range(0, n, 2048):
        loss = F.binary_cross_entropy_with_logits(_logits64(p, stamps[a:a + 2048]), labels[a:a + 2048].double(), reduction="sum") / n
        loss.backward()
        total += loss.detach()
    return dict(grad={k: v.grad.reshape(-1) for k, v in p.items()}, loss=total.reshape(1))
