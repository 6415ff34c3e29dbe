"""Performance cases of the screening library: the calls a screening program
makes, through the package's public entry points, over the sizes it makes
them at.

A case is a dict of plain values; its ``kind`` says which call it stands for:

  screen   boxes and candidate pairs of one scene (whole-scene tree or a static
           decomposition), the list left on the device or brought to the host
  narrow   collision witnesses inside a screen's candidate list
  refine   every collision witness by adaptive refinement (or, with eps_s > 0,
           the spans of its continuous-time variant)
  batch    many independent scenes screened as one
  train    the step network's training gradient over one minibatch

``prepare`` makes what a program holds before the call (the scene with its
elements, a trained step network, the arrays its results go to, sized for the
workload with some room), ``run`` is one call.  Result arrays are returned
whole: the rows past a list's end keep their -1.
"""
import math

import numpy as np
import torch

import paper_1901_10475_gb300 as scd
import population as P
from paper_1901_10475_gb300.stepnet import StepNet

# the tuning that the autotuner picks for the slab-octant screen of the 24 h
# catalog, with the find sequence replayed as one graph
SLAB_TUNING = dict(morton_bits=10, time_scale=4.0, space_warp=1, use_graph=1)


def listed():
    return [
        # the smallest call: 512 objects in low orbits over 100 minutes at a
        # fixed 10 s step, elements in from the host, the list out as numpy;
        # a service that answers single questions runs at this latency
        dict(name="screen_512_host", kind="screen", pop="leo", n=512, minutes=100, mode="speed",
             step="fixed", fraction=10.0, decomp="none", cells=0, out="numpy"),
        # a regional subset over two hours (odd sizes), re-screened as its
        # elements change: between launch-bound and throughput-bound
        dict(name="screen_3001_2h", kind="screen", pop="catalog", n=3001, minutes=127,
             mode="speed", step="period", fraction=100.0, decomp="none", cells=0, out="device"),
        # the headline workload: the whole catalog over 24 h
        dict(name="screen_16848_24h", kind="screen", pop="catalog", n=16848, minutes=1440,
             mode="speed", step="period", fraction=100.0, decomp="none", cells=0, out="device"),
        # the same with the tighter boxes of interval arithmetic
        dict(name="screen_16848_24h_interval", kind="screen", pop="catalog", n=16848,
             minutes=1440, mode="interval", step="period", fraction=100.0, decomp="none", cells=0,
             out="device"),
        # host to host: pinned elements in, the whole pair list out into
        # pinned memory, as a program without a GPU consumer takes it
        dict(name="screen_6007_24h_host", kind="screen", pop="catalog", n=6007, minutes=1440,
             mode="speed", step="period", fraction=100.0, decomp="none", cells=0, out="pinned"),
        # 100k-class populations with dense shells, steps from the network
        dict(name="screen_20011_24h_learned", kind="screen", pop="shells", n=20011, minutes=1440,
             mode="interval", step="learned", fraction=140.0, decomp="none", cells=0,
             out="device"),
        # the static decomposition: 16 tick slabs x 8 octants, band steps,
        # replayed as one graph
        dict(name="screen_16848_24h_slabs", kind="screen", pop="catalog", n=16848, minutes=1440,
             mode="speed", step="band", fraction=0.0, decomp="slabs", cells=16, out="device"),
        # the first witness over the whole catalog's candidates
        dict(name="narrow_16848_24h", kind="narrow", pop="catalog", n=16848, minutes=1440,
             mode="speed", step="period", fraction=100.0),
        # adaptive refinement, small (a service's latency) and the catalog
        dict(name="refine_512", kind="refine", pop="leo", n=512, minutes=100, mode="speed",
             eps_s=0.0),
        dict(name="refine_16848_24h", kind="refine", pop="catalog", n=16848, minutes=1440,
             mode="speed", eps_s=0.0),
        # independent scenes of uneven size and horizon in one call
        dict(name="batch_11", kind="batch", scenes=11, lo=1000, hi=8000, hours_lo=6, hours_hi=36),
        # one minibatch of the step network's training
        dict(name="train_4096", kind="train", n=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["screen", "screen", "screen", "screen", "narrow", "refine", "refine",
                       "batch", "train"])
    if kind == "train":
        return dict(kind=kind, n=_log_int(rng, 200, 16384))
    if kind == "batch":
        lo = _log_int(rng, 300, 2000)
        return dict(kind=kind, scenes=rng.randint(2, 11), lo=lo, hi=rng.randint(2 * lo, 8000),
                    hours_lo=rng.randint(2, 8), hours_hi=rng.randint(9, 36))
    pop = rng.choice(["leo", "catalog", "catalog"])
    n = _log_int(rng, 150, 2000) if pop == "leo" else _log_int(rng, 300, 16848)
    c = dict(kind=kind, pop=pop, n=n, minutes=_log_int(rng, 30, 1440 if pop != "leo" else 200),
             mode=rng.choice(["speed", "speed", "interval"]))
    if kind == "refine":
        # the continuous variant's work grows with the crowding: small scenes
        c["eps_s"] = rng.choice([0.5, 1.0, 2.0]) if pop == "leo" and n < 800 else 0.0
        return c
    if pop == "leo":
        c.update(step="fixed", fraction=float(rng.randint(5, 60)))
    else:
        c.update(step="period", fraction=float(rng.randint(80, 200)))
    if kind == "narrow":
        return c
    c.update(decomp="none", cells=0, out=rng.choice(["device", "device", "pinned", "numpy"]))
    if pop == "catalog":
        c["step"] = rng.choice(["period", "period", "period", "band", "learned"])
        c["decomp"] = rng.choice(["none", "none", "none", "slabs", "bands"])
        if c["decomp"] != "none":
            c["cells"] = rng.randint(2, 16)
            c["out"] = "device"
    if c["out"] == "numpy":  # small lists, as a script takes them
        c["n"], c["minutes"] = min(n, 1000), min(c["minutes"], 200)
    return c


def _elements(case, seed):
    horizon = 60.0 * case["minutes"]
    s = P.SEED_BASE + 1000 + seed
    if case["pop"] == "leo":
        return P.uniform_leo(case["n"], seed=s), horizon
    return P.catalog_mixture(case["n"], seed=s, horizon_s=horizon,
                             dense_shells=case["pop"] == "shells"), horizon


def _step_params(fraction, seed):
    """Step-network parameters that give P / fraction with somewhat shorter
    steps in crowded shells, and small trained-like weights elsewhere."""
    nin, hid = scd.SCD_STEPNET_IN, scd.SCD_STEPNET_HIDDEN
    g = np.random.Generator(np.random.Philox(seed))
    w1 = g.normal(0.0, 0.01, (nin, hid))
    w2 = g.normal(0.0, 0.01, (hid, hid))
    w3 = g.normal(0.0, 0.01, hid)
    w1[:, :2] = 0.0
    w2[:, :2] = 0.0
    w1[6, 0] = w1[7, 1] = 1.0  # log(P / 1 h) and the crowding pass through
    w2[0, 0] = w2[1, 1] = 1.0
    w3[0], w3[1] = 1.0, -0.03
    b3 = math.log(3600.0 / fraction) + 0.15
    return np.concatenate([w1.ravel(), np.zeros(hid), w2.ravel(), np.zeros(hid), w3,
                           [b3]]).astype(np.float32)


def _mode(case):
    return scd.SCD_BOX_INTERVAL if case["mode"] == "interval" else scd.SCD_BOX_SPEED


def _policy(case, seed, keep):
    if case["step"] == "fixed":
        return scd.make_step_policy(scd.SCD_STEP_FIXED, fixed_ticks=int(case["fraction"]))
    if case["step"] == "band":
        edges, fractions = P.band_table_config3()
        return scd.make_step_policy(scd.SCD_STEP_BAND_TABLE, band_edges_km=edges,
                                    band_fractions=fractions)
    if case["step"] == "learned":
        keep["net"] = StepNet(seed=seed)
        keep["net"].params = _step_params(case["fraction"], seed)
        return keep["net"].policy()
    return scd.make_step_policy(scd.SCD_STEP_PERIOD_FRACTION, period_fraction=case["fraction"])


def prepare(case, seed):
    st = dict(case=case)
    if case["kind"] == "train":
        x, t, params = _train_inputs(case, seed)
        st["net"] = StepNet(seed=1)
        st["net"].params = params
        st["x"], st["t"] = torch.as_tensor(x, device="cuda"), torch.as_tensor(t, device="cuda")
        return st
    if case["kind"] == "batch":
        scenes, hours = _batch(case, seed)
        st["scene"] = scd.BatchScene(scenes, hours, 1.0, mode=scd.SCD_BOX_INTERVAL)
        st["out"] = torch.full((_room(_batch_work(case)[0]), 4), -1, dtype=torch.int32,
                               device="cuda")
        return st
    els, horizon = _elements(case, seed)
    if case["kind"] == "refine":
        st["scene"] = scd.Scene(els, horizon, 1.0, mode=_mode(case))
        st["host"] = np.full((65536 + 8 * case["n"], 6 if case["eps_s"] > 0.0 else 3), -1, np.int32)
        st["rounds"] = np.full(64, -1, np.int64)
        return st
    st["scene"] = scd.Scene(els, horizon, 1.0, _policy(case, seed, st), mode=_mode(case))
    if case["kind"] == "narrow":
        # the candidates of the scene's own screen
        st["pairs"] = st["scene"].build_boxes().find_pairs_device()
        st["out"] = torch.full((2, _room(_scene_work(case)[0])), -1, dtype=torch.int32,
                               device="cuda")
        return st
    st["decomp"] = None
    if case["decomp"] == "slabs":
        st["decomp"] = (scd.SCD_DECOMP_SLAB_OCT, 0, case["cells"])
        st["scene"].set_tuning(dict(st["scene"].tuning(), **SLAB_TUNING))
    elif case["decomp"] == "bands":
        st["decomp"] = (scd.SCD_DECOMP_ALT_BANDS, case["cells"], 0)
    if case["out"] != "device":
        st["els"] = torch.as_tensor(els).pin_memory().numpy()
    shape = (_room(_scene_work(case)[0]), 4)
    if case["out"] == "device":
        st["out"] = torch.full(shape, -1, dtype=torch.int32, device="cuda")
    else:
        host = torch.full(shape, -1, dtype=torch.int32)
        st["out"] = (host.pin_memory() if case["out"] == "pinned" else host).numpy()
    return st


def _keep(out, rows):
    """A result that belongs to the scene, or a new one, into the program's array."""
    if len(rows) > len(out):
        raise RuntimeError("%d rows, room for %d" % (len(rows), len(out)))
    out[:len(rows)] = rows
    return out


def run(st):
    case = st["case"]
    if case["kind"] == "train":
        loss, grad = st["net"].grad(st["x"], st["t"])
        return dict(loss=loss, grad=grad)
    sc = st["scene"]
    if case["kind"] == "narrow":
        first, count = st["out"]
        m = len(st["pairs"])
        if m > len(first):
            raise RuntimeError("%d candidates, room for %d" % (m, len(first)))
        w = scd.scd_narrow_phase(sc.handle, st["pairs"].data_ptr() if m else 0, m,
                                 first.data_ptr(), count.data_ptr())
        return dict(first=first, count=count, earliest=w or (-1, -1, -1))
    if case["kind"] == "refine":
        sc.build_boxes()
        if case["eps_s"] > 0.0:
            found, rounds = sc.refine_continuous(case["eps_s"])
        else:
            found, rounds = sc.refine_witnesses()
        # the records' words: i, j, t of a witness, i, j, t0, t1 of a span
        words = found.view(np.int32).reshape(len(found), st["host"].shape[1])
        return dict(found=_keep(st["host"], words), rounds=_keep(st["rounds"], rounds))
    if case["kind"] == "batch":
        sc.build_boxes()
        pairs = _keep(st["out"], sc.find_pairs_device())
        return dict(pairs=pairs, offsets=scd.scd_batch_scene_offsets(sc.handle, sc.n_scenes))
    if case["out"] != "device":
        sc.set_elements(st["els"])
    sc.build_boxes()
    if case["out"] == "device":
        return _keep(st["out"], sc.find_pairs_device(st["decomp"]))
    if case["out"] == "numpy":
        pairs = sc.find_pairs(st["decomp"])
        return _keep(st["out"], pairs.view(np.int32).reshape(len(pairs), 4))
    scd.scd_find_pairs_into(sc.handle, st["out"].view(scd.PAIR_DTYPE).reshape(-1), st["decomp"])
    return st["out"]


def _batch(case, seed):
    g = np.random.Generator(np.random.Philox(P.SEED_BASE + 3000 + seed))
    # the sizes and horizons belong to the case; the seed makes the orbits
    h = np.random.Generator(np.random.Philox(case["scenes"] * 100003 + case["lo"]))
    sizes = np.exp(h.uniform(math.log(case["lo"]), math.log(case["hi"]), case["scenes"]))
    hours = h.integers(case["hours_lo"], case["hours_hi"] + 1, case["scenes"])
    scenes = [P.catalog_mixture(int(m), seed=int(g.integers(1 << 40)), horizon_s=3600.0 * int(hr))
              for m, hr in zip(sizes, hours)]
    return scenes, [3600.0 * int(hr) for hr in hours]


def _train_inputs(case, seed):
    """Features of a catalog's objects, the log of a per-object best step [s]
    (a fraction between P/70 and P/280), and untrained parameters."""
    els = P.catalog_mixture(case["n"], seed=P.SEED_BASE + 2000 + seed)
    a, e, inc = els[:, 0], els[:, 1], els[:, 2]
    period = 2.0 * math.pi * np.sqrt(a ** 3 / P.MU)
    order = np.sort(a)
    near = (np.searchsorted(order, a + 50.0, "right") - np.searchsorted(order, a - 50.0, "left"))
    x = np.stack([np.log(a / P.RE), e, np.sin(inc), np.cos(inc),
                  np.log(np.maximum(a * (1.0 - e) - P.RE, 1.0) / 100.0),
                  np.log(np.maximum(a * (1.0 + e) - P.RE, 1.0) / 100.0),
                  np.log(period / 3600.0), np.log1p(near - 1.0)], 1)
    g = np.random.Generator(np.random.Philox(P.SEED_BASE + 4000 + seed))
    t = np.log(period / np.exp(g.uniform(math.log(70.0), math.log(280.0), len(els))))
    nin, hid = scd.SCD_STEPNET_IN, scd.SCD_STEPNET_HIDDEN
    w = [g.uniform(-1.0, 1.0, m) * math.sqrt(6.0 / f)
         for m, f in ((nin * hid, nin), (hid * hid, hid), (hid, 2 * hid))]
    params = np.concatenate([w[0], g.normal(0, 0.1, hid), w[1], g.normal(0, 0.1, hid), w[2],
                             [5.0]])
    return x.astype(np.float32), t.astype(np.float32), params.astype(np.float32)


def _boxes(els, horizon, fraction):
    period = 2.0 * math.pi * np.sqrt(els[:, 0] ** 3 / P.MU)
    k = np.maximum(np.floor(period / fraction), 1.0)
    return float(np.sum(np.ceil((horizon + 1.0) / k)))


# Candidate pairs of one screen per object pair and hour: the catalog at
# P / 100 with each kind of box, and the low-orbit shell at 10 s steps
# (measured; the lists go with the square of the box size)
_PAIRS = {("catalog", "speed"): 0.048, ("catalog", "interval"): 0.0076,
          ("shells", "interval"): 0.0086, ("leo", "speed"): 0.00046, ("leo", "interval"): 0.00040}


def _room(pairs):
    return int(1.3 * pairs) + 65536


# FP64 operations of one box: a Kepler solve, the position, the faces
_OPS = 60.0


def _scene_work(case):
    els, horizon = _elements(case, 0)
    n, hours = case["n"], case["minutes"] / 60.0
    step = case.get("step", "period")
    f = {"fixed": None, "band": 125.0, "period": case.get("fraction", 100.0),
         "learned": 140.0}[step]
    if f is None:
        scale, boxes = (case["fraction"] / 10.0) ** 2, n * math.ceil((horizon + 1.0) / case["fraction"])
    else:
        scale, boxes = (100.0 / f) ** 2, _boxes(els, horizon, f)
    pairs = 0.5 * n * n * hours * scale * _PAIRS[case["pop"], case["mode"]]
    return pairs, boxes


def _batch_work(case):
    scenes, horizons = _batch(case, 0)
    pairs = sum(0.5 * len(e) ** 2 * (h / 3600.0) * _PAIRS["catalog", "interval"]
                for e, h in zip(scenes, horizons))
    boxes = sum(_boxes(e, h, 100.0) for e, h in zip(scenes, horizons))
    return pairs, boxes, sum(map(len, scenes))


def work(case):
    if case["kind"] == "train":
        # forward, and the gradient with respect to weights and activations;
        # features and targets in, weights in, gradient out
        macs = 8 * 64 + 64 * 64 + 64
        return dict(bytes=case["n"] * 36 + 2 * 4 * scd.SCD_STEPNET_PARAMS,
                    flops=6.0 * macs * case["n"])
    if case["kind"] == "batch":
        pairs, boxes, n = _batch_work(case)
        return dict(bytes=56 * n + 16 * pairs, flops=2 * _OPS * boxes)
    per_box = _OPS * (2 if case["mode"] == "interval" else 1)
    if case["kind"] == "refine":
        # the boxes of one level that proves most intervals free (about ten
        # seconds of motion); the witnesses are few
        els, horizon = _elements(case, 0)
        return dict(bytes=56 * case["n"], flops=per_box * _boxes(els, horizon, 256.0))
    pairs, boxes = _scene_work(case)
    if case["kind"] == "narrow":
        # candidates in, first tick and count out; two positions a candidate
        return dict(bytes=56 * case["n"] + 24 * pairs, flops=2 * _OPS * pairs)
    return dict(bytes=56 * case["n"] + 16 * pairs, flops=per_box * boxes)


def exact(case, seed):
    """The training gradient in 64 bits; every other output is whole numbers."""
    if case["kind"] != "train":
        return None
    nin, hid = scd.SCD_STEPNET_IN, scd.SCD_STEPNET_HIDDEN
    x, t, p = (torch.from_numpy(v) for v in _train_inputs(case, seed))
    x, t = x.double(), t.double()
    cut = np.cumsum([0, nin * hid, hid, hid * hid, hid, hid, 1])
    part = [p[a:b] for a, b in zip(cut[:-1], cut[1:])]
    # the network's weights are BF16 by its definition, its biases FP32
    part = [(q.bfloat16() if k in (0, 2, 4) else q).double().requires_grad_()
            for k, q in enumerate(part)]
    w1, b1, w2, b2, w3, b3 = part
    h1 = torch.relu(x @ w1.view(nin, hid) + b1)
    h2 = torch.relu(h1 @ w2.view(hid, hid) + b2)
    loss = torch.mean((h2 @ w3 + b3 - t) ** 2)
    loss.backward()
    return dict(loss=float(loss.detach()), grad=torch.cat([q.grad for q in part]))
