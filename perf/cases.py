"""Performance cases: the calls a user of the ray tracer and of its learned
surrogate makes, at the sizes of the repository's configurations and tests.

  links          compute_paths, paths(), cir(), freq_response() for a set of
                 receivers. `links_tiny` is the smallest call (one box, one
                 receiver; launches and read-backs count), `links_city` the
                 city configuration (4802 triangles, 1000 receivers, 1e6 rays,
                 1024 subcarriers).
  labels         surrogate.tracer_labels: batches of transmitters, each with
                 its own receivers, to (has path, gain dB) pairs.
  coverage       coverage_map: one sector over the city, and 64 rooftop
                 transmitters of 1e7 rays each at depth 5 in one launch.
  coverage_vjp   coverage_map_backward: the orientation gradient of a map.
  gradient       one calibration step through the autograd functions: forward
                 CIR and H(f), NMSE loss, backward to materials and pose.
  freq           rt_freq_response_paths over a dense path list (channels from
                 elsewhere), where H(f) is arithmetic and not stores.
  scattering     scattering_gain: first-order diffuse scattering, every ray's
                 hit against every receiver.
  diffraction_map  coverage_map_diffraction: every cell against every wedge.
  infer          Surrogate.infer, the network that stands in for the tracer.
  train          Surrogate.train_step at the batch size the surrogate is
                 trained with. The learning rate is 0 (the first step of a
                 linear warm-up), so that every pass is the same step; the
                 gradients are what is compared.

Each state holds its own Tracer or Surrogate with the scene loaded and the
devices set, as a user's program does; the scene, the devices and all values
come from the seed. Shapes, depths, antennas and counts come from the case.
The number of paths of `links` depends on the places, so there the buildings
and the sites come from the case ("place"), and the seed gives the materials,
the orientations and the order of the receivers.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2303_11103_gb300 import learning as LG
from paper_2303_11103_gb300 import rt
from paper_2303_11103_gb300 import scenes as S
from paper_2303_11103_gb300 import surrogate as SG

FC = 3.5e9
SPACING = 30e3
ANTENNAS = {"iso": S.V_ISO, "dipole": S.Antenna(S.ANT_DIPOLE, (0.0,)), "sector": S.TR38901_V,
            "sector_dual": S.TR38901_VH}


def listed():
    return [
        # the tiny configuration with a visible receiver: latency of the smallest call
        {"name": "links_tiny", "kind": "links", "n_side": 0, "n_tx": 1, "n_rx": 1, "rays": 10_000, "depth": 2,
         "sc": 64, "place": 1, "tx_ant": "iso", "rx_ant": "iso"},
        # the city configuration: link-level channels of a sector's 1000 users
        {"name": "links_city", "kind": "links", "n_side": 20, "n_tx": 1, "n_rx": 1000, "rays": 1_000_000, "depth": 3,
         "sc": 1024, "place": 1, "tx_ant": "sector_dual", "rx_ant": "iso"},
        # training labels of the surrogate: one batch of 32 sites x 250 receivers
        {"name": "labels_32x250", "kind": "labels", "n_side": 20, "n_tx": 32, "n_rx": 250, "rays": 200_000, "depth": 3},
        # coverage of one sector, 1 m cells
        {"name": "coverage_city", "kind": "coverage", "n_side": 20, "n_tx": 1, "rays": 1_000_000, "depth": 3,
         "nx": 500, "ny": 500, "cell": 1.0, "tx_ant": "sector_dual", "port": 0},
        # the batched configuration: network planning over 64 rooftops, the largest call
        {"name": "coverage_batch64", "kind": "coverage", "n_side": 20, "n_tx": 64, "rays": 10_000_000, "depth": 5,
         "nx": 500, "ny": 500, "cell": 1.0, "tx_ant": "sector", "port": 0},
        # one ascent step of an antenna's orientation
        {"name": "coverage_vjp_city", "kind": "coverage_vjp", "n_side": 20, "n_tx": 1, "rays": 1_000_000, "depth": 3,
         "nx": 500, "ny": 500, "cell": 1.0, "tx_ant": "sector_dual", "port": 0},
        # the differentiation configuration: 8 materials, 256 receivers, 128 subcarriers
        {"name": "gradient_256rx", "kind": "gradient", "n_side": 20, "n_mat": 8, "n_rx": 256, "rays": 1_000_000,
         "depth": 3, "sc": 128, "tx_ant": "sector_dual", "rx_ant": "iso"},
        # H(f) of 1000 links with 64 paths each, 2 x 2 ports
        {"name": "freq_dense", "kind": "freq", "pairs": 1000, "mean_paths": 64, "ports": 4, "sc": 1024,
         "uniform": True},
        # diffuse scattering to the city's receivers
        {"name": "scattering_city", "kind": "scattering", "n_side": 20, "n_tx": 1, "n_rx": 1000, "rays": 100_000,
         "coeff": 0.3, "alpha": -1, "tx_ant": "sector_dual", "rx_ant": "iso"},
        # the diffracted part of the city's coverage map
        {"name": "diffraction_map_city", "kind": "diffraction_map", "n_side": 20, "n_tx": 1, "nx": 500, "ny": 500,
         "cell": 1.0, "tx_ant": "sector_dual", "port": 0},
        # a million surrogate queries
        {"name": "infer_1M", "kind": "infer", "n": 1_000_000, "freqs": 32, "width": 256, "hidden": 8},
        # one optimiser step of the surrogate
        {"name": "train_16384", "kind": "train", "n": 16384, "freqs": 32, "width": 256, "hidden": 8},
    ]


# ------------------------------------------------------------------ drawn cases
def _log(rng, lo, hi):
    """An integer spread evenly over the logarithm of [lo, hi]."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _size(n_side):
    return 25.0 * n_side if n_side else 200.0


def draw(rng):
    kind = rng.choice(["links", "labels", "coverage", "coverage_vjp", "gradient", "freq", "scattering",
                       "diffraction_map", "infer", "train"])
    # from 250 m on, only the ground is larger than the buildings
    side = _log(rng, 10, 24)
    if kind == "links":
        side = _log(rng, 4, 24)
        depth = rng.randint(1, 4)
        return {"kind": kind, "n_side": side, "n_tx": rng.randint(1, 4), "n_rx": _log(rng, 1, 2000),
                "rays": _log(rng, 1000, 1_000_000), "depth": depth, "sc": _log(rng, 1, 2048), "place": rng.randint(1, 999),
                "tx_ant": rng.choice(sorted(ANTENNAS)), "rx_ant": rng.choice(sorted(ANTENNAS))}
    if kind == "labels":
        return {"kind": kind, "n_side": side, "n_tx": rng.randint(2, 64), "n_rx": _log(rng, 10, 500),
                "rays": _log(rng, 10_000, 200_000), "depth": rng.randint(1, 3)}
    if kind in ("coverage", "coverage_vjp"):
        n_tx = _log(rng, 1, 32) if kind == "coverage" else rng.randint(1, 4)
        nx, ny = rng.randint(20, 500), rng.randint(20, 500)
        return {"kind": kind, "n_side": side, "n_tx": n_tx, "rays": _log(rng, 1000, 2_000_000),
                "depth": rng.randint(0, 5), "nx": nx, "ny": ny, "cell": _size(side) / max(nx, ny),
                "tx_ant": rng.choice(sorted(ANTENNAS)), "port": 0}
    if kind == "gradient":
        return {"kind": kind, "n_side": side, "n_mat": rng.randint(2, 12), "n_rx": _log(rng, 64, 2000),
                "rays": _log(rng, 20_000, 1_000_000), "depth": rng.randint(1, 3), "sc": _log(rng, 8, 512),
                "tx_ant": "sector_dual", "rx_ant": rng.choice(["iso", "sector_dual"])}
    if kind == "freq":
        return {"kind": kind, "pairs": _log(rng, 2, 2000), "mean_paths": _log(rng, 1, 100),
                "ports": rng.choice([1, 2, 4]), "sc": _log(rng, 1, 2048), "uniform": rng.random() < 0.7}
    if kind == "scattering":
        return {"kind": kind, "n_side": side, "n_tx": rng.randint(1, 3), "n_rx": _log(rng, 1, 1500),
                "rays": _log(rng, 1000, 200_000), "coeff": round(rng.uniform(0.1, 0.9), 3),
                "alpha": rng.choice([-1, -1, 4]), "tx_ant": rng.choice(sorted(ANTENNAS)),
                "rx_ant": rng.choice(sorted(ANTENNAS))}
    if kind == "diffraction_map":
        side = min(side, 20)
        nx, ny = rng.randint(20, 400), rng.randint(20, 400)
        return {"kind": kind, "n_side": side, "n_tx": rng.randint(1, 2), "nx": nx, "ny": ny,
                "cell": _size(side) / max(nx, ny), "tx_ant": rng.choice(sorted(ANTENNAS)), "port": 0}
    if kind == "infer":
        return {"kind": kind, "n": _log(rng, 1, 4_000_000), "freqs": rng.choice([32, 64]),
                "width": rng.choice([64, 128, 256]), "hidden": rng.randint(2, 8)}
    return {"kind": "train", "n": 128 * _log(rng, 1, 256), "freqs": rng.choice([16, 32]),
            "width": rng.choice([64, 128, 256]), "hidden": rng.randint(2, 8)}


# ----------------------------------------------------------------------- inputs
def _city(c, seed):
    if c["n_side"] == 0:
        return S.tiny_scene()
    return S.city_scene(n_side=c["n_side"], size=_size(c["n_side"]), seed=seed % 9973, n_materials=c.get("n_mat", 0),
                        mat_seed=seed % 9973 + 1)


def _streets(scene, n, rng, half, taller_than=0.0):
    """n points uniform over [-half, half]^2 outside every building of more than
    the given height (a wider square while a small city has too few)."""
    f = scene.footprints
    f = f[f[:, 4] > taller_than]
    out = np.zeros((0, 2))
    while len(out) < n:
        p = rng.uniform(-half, half, (2 * (n - len(out)) + 64, 2))
        half *= 1.02
        x, y = p[:, :1], p[:, 1:]
        inside = ((x > f[:, 0] - 0.5) & (x < f[:, 1] + 0.5) & (y > f[:, 2] - 0.5) & (y < f[:, 3] + 0.5)).any(1)
        out = np.concatenate([out, p[~inside]])
    return out[:n]


def _transmitters(c, scene, rng):
    """30 m masts over streets, or (many) 25 to 60 m sites not inside a taller building."""
    half, n = 0.48 * _size(c["n_side"]), c["n_tx"] if "n_tx" in c else 1
    z = np.full(n, 30.0) if n <= 4 else rng.uniform(25.0, 60.0, n)
    xy = _streets(scene, n, rng, 0.6 * half) if n <= 4 else np.concatenate(
        [_streets(scene, 1, rng, half, taller_than=h - 1.0) for h in z])
    ypr = np.stack([rng.uniform(-np.pi, np.pi, n), np.full(n, 0.1), np.zeros(n)], 1)
    return np.concatenate([xy, z[:, None]], 1).astype(np.float32), ypr.astype(np.float32)


def _receivers(c, scene, rng):
    n = c["n_rx"]
    if c["n_side"] == 0:   # near the box's wall, where line of sight, ground and wall paths exist
        xy = np.stack([rng.uniform(-80.0, -70.0, n), rng.uniform(-5.0, 5.0, n)], 1)
    else:
        xy = _streets(scene, n, rng, 0.48 * _size(c["n_side"]))
    pos = np.concatenate([xy, np.full((n, 1), 1.5)], 1).astype(np.float32)
    return pos, rng.uniform(-0.2, 0.2, (n, 3)).astype(np.float32)


def _tracer(c, seed, receivers=True):
    place = c.get("place", seed)
    rng = np.random.default_rng(place)
    scene = _city(c, place)
    own = np.random.default_rng(seed + 1)   # what does not change the number of paths
    if "place" in c:
        scene.materials = (scene.materials * own.uniform(0.8, 1.25, scene.materials.shape)).astype(np.float32)
    tr = rt.Tracer(0, FC)
    tr.load_scene(scene)
    if c["n_side"] == 0:
        tx = (np.array([[-60.0, 0.0, 25.0]]) + rng.uniform(-2.0, 2.0, (1, 3))).astype(np.float32)
        ypr = rng.uniform(-0.2, 0.2, (1, 3)).astype(np.float32)
    else:
        tx, ypr = _transmitters(c, scene, rng)
    if "place" in c:
        ypr = (ypr + own.uniform(-0.5, 0.5, ypr.shape)).astype(np.float32)
    tr.set_tx(tx, ypr, ANTENNAS[c.get("tx_ant", "iso")])
    if receivers:
        pos, rypr = _receivers(c, scene, rng)
        if "place" in c:
            pos = pos[own.permutation(len(pos))]
        tr.set_rx(pos, rypr, ANTENNAS[c.get("rx_ant", "iso")])
    else:
        tr.set_rx(np.zeros((1, 3), np.float32), np.zeros((1, 3), np.float32), S.V_ISO)
    return tr, scene, rng


def _grid(c):
    half = 0.5 * _size(c["n_side"])
    return dict(x0=-half, y0=-half, cell=c["cell"], nx=c["nx"], ny=c["ny"], h=1.5)


def _subcarriers(n):
    return (torch.arange(n, dtype=torch.float64, device="cuda") - n // 2) * SPACING


def _path_list(c, seed):
    off, a, tau = S.dense_path_list(c["pairs"], c["mean_paths"], c["ports"], seed=seed)
    K = c["sc"]
    if c["uniform"]:
        freqs = (np.arange(K) - K // 2) * SPACING
    else:   # occupied resource blocks only: sorted, uneven
        freqs = np.sort(np.random.default_rng(seed + 1).choice(2 * K, K, replace=False) - K) * SPACING
    return off, a, tau, freqs.astype(np.float64)


def _layer_dims(c):
    d = [(c["width"], 2 * c["freqs"] if k == 0 else c["width"]) for k in range(c["hidden"])]
    return d + [(2, c["width"])]


BOX = (np.array([-240.0, -240.0, 10.0, -240.0, -240.0, 1.5]), np.array([240.0, 240.0, 65.0, 240.0, 240.0, 2.5]))


def _network(c, seed):
    """Parameters of a network (float32, in the order of Surrogate.params()), and queries in its box."""
    g = torch.Generator(device="cuda").manual_seed(seed)

    def uniform(*shape):
        return 2.0 * torch.rand(shape, generator=g, device="cuda") - 1.0

    parts = []
    for out, inp in _layer_dims(c):
        parts += [uniform(out * inp) * math.sqrt(6.0 / inp) * (1.0 if out > 2 else 0.5), 0.1 * uniform(out)]
    parts.append(torch.randn(6 * c["freqs"], generator=g, device="cuda"))
    lo, hi = (torch.as_tensor(v, dtype=torch.float32, device="cuda") for v in BOX)
    x = lo + (hi - lo) * torch.rand((c["n"], 6), generator=g, device="cuda")
    has = (torch.rand(c["n"], generator=g, device="cuda") < 0.3).float()
    gain = -140.0 + 70.0 * torch.rand(c["n"], generator=g, device="cuda")
    target = torch.stack([has, torch.where(has > 0, gain, torch.full_like(gain, -400.0))], 1)
    return torch.cat(parts).float(), x.contiguous(), target.contiguous()


def prepare(case, seed):
    c, kind = case, case["kind"]
    st = {"case": c}
    if kind == "links":
        st["tracer"], _, _ = _tracer(c, seed)
        st["freqs"] = _subcarriers(c["sc"])
    elif kind == "labels":
        scene = _city(c, seed)
        rng = np.random.default_rng(seed)
        half = 0.48 * _size(c["n_side"])
        z = rng.uniform(25.0, 60.0, c["n_tx"])
        xy = np.concatenate([_streets(scene, 1, rng, half, taller_than=h - 1.0) for h in z])
        st["tx"] = np.concatenate([xy, z[:, None]], 1).astype(np.float32)
        rx = _streets(scene, c["n_tx"] * c["n_rx"], rng, half)
        rx = np.concatenate([rx, np.full((len(rx), 1), 1.5)], 1)
        st["rx"] = rx.reshape(c["n_tx"], c["n_rx"], 3).astype(np.float32)
        st["tracer"] = rt.Tracer(0, FC)
        st["tracer"].load_scene(scene)
    elif kind in ("coverage", "coverage_vjp", "diffraction_map"):
        st["tracer"], _, rng = _tracer(c, seed, receivers=False)
        st["grid"] = _grid(c)
        if kind == "coverage_vjp":
            g = torch.Generator(device="cuda").manual_seed(seed)
            st["grad"] = torch.rand((c["n_tx"], c["ny"], c["nx"]), generator=g, device="cuda")
    elif kind == "gradient":
        tr, _, rng = _tracer(c, seed)
        tr.compute_paths(c["depth"], c["rays"])
        st["tracer"], st["freqs"] = tr, _subcarriers(c["sc"])
        a, tau = tr.cir()
        H = tr.freq_response(a, tau, st["freqs"])
        g = torch.Generator(device="cuda").manual_seed(seed)
        noise = torch.randn(H.shape + (2,), generator=g, device="cuda")
        st["H_ref"] = 1.1 * H + 0.1 * H.abs() * torch.view_as_complex(noise)
        m = tr._mats
        st["leaves"] = [m[:, 0] * 1.2, m[:, 1] * 0.8, tr._tx_pos.clone(), tr._tx_ypr.clone()]
    elif kind == "freq":
        off, a, tau, freqs = _path_list(c, seed)
        st["tracer"] = rt.Tracer(0, FC)
        st["off"] = torch.as_tensor(off, device="cuda")
        st["a"] = torch.view_as_real(torch.as_tensor(a, device="cuda")).contiguous()
        st["tau"] = torch.as_tensor(tau, device="cuda")
        st["freqs"] = torch.as_tensor(freqs, device="cuda")
    elif kind == "scattering":
        tr, _, _ = _tracer(c, seed)
        tr.set_scattering([c["coeff"]] * tr.n_mat)
        tr.set_scattering_pattern([c["alpha"]] * tr.n_mat)
        st["tracer"] = tr
    else:
        p, st["x"], st["target"] = _network(c, seed)
        st["net"] = rt.Surrogate(BOX[0], BOX[1], n_freq=c["freqs"], width=c["width"], n_hidden=c["hidden"])
        st["net"].set_params(p)
    return st


# ------------------------------------------------------------------------- runs
def run(state):
    c, tr = state["case"], state.get("tracer")
    kind = c["kind"]
    if kind == "links":
        tr.compute_paths(c["depth"], c["rays"])
        out = tr.paths()
        a, tau = tr.cir()
        return dict(out, a=a, tau=tau, H=tr.freq_response(a, tau, state["freqs"]))
    if kind == "labels":
        x, t = SG.tracer_labels(tr, state["tx"], state["rx"], c["rays"], c["depth"])
        return {"x": x, "target": t}
    if kind == "coverage":
        gain, hits = tr.coverage_map(state["grid"], c["depth"], c["rays"], c["port"])
        return {"gain": gain, "hits": hits}
    if kind == "coverage_vjp":
        return tr.coverage_map_backward(state["grid"], c["depth"], c["rays"], state["grad"], c["port"])
    if kind == "diffraction_map":
        return tr.coverage_map_diffraction(state["grid"], c["port"])
    if kind == "gradient":
        leaves = [v.detach().requires_grad_(True) for v in state["leaves"]]
        a, tau = rt.CIR.apply(tr, *leaves)
        H = rt.FreqResponse.apply(tr, a, tau, state["freqs"])
        loss = LG.nmse(H, state["H_ref"])
        loss.backward()
        return {"loss": loss.detach(), "H": H.detach(), "grads": [v.grad for v in leaves]}
    if kind == "freq":
        H = torch.empty((c["pairs"], c["ports"], c["sc"], 2), dtype=torch.float32, device="cuda")
        tr.sync_stream()
        rt.rt_freq_response_paths(tr.ctx, state["off"], c["ports"], state["a"], state["tau"], state["freqs"], H)
        return H
    if kind == "scattering":
        return tr.scattering_gain(c["rays"])
    if kind == "infer":
        return state["net"].infer(state["x"])
    loss = torch.zeros(1, device="cuda")
    state["net"].train_step(state["x"], state["target"], 0.0, loss)
    return {"loss": loss, "grads": state["net"].grads()}


# ------------------------------------------------------------------------- work
def work(case):
    """Least bytes and operations of one pass. A traced ray segment takes at
    least one path from the root of a binary tree over the triangles to its
    hit (2 box tests of 11 operations per level) and one triangle test (35);
    a visibility test the same. Bytes: each input read and each output
    written once (the path list of `links` depends on the scene and is left
    out, H(f) is written for every pair)."""
    c, kind = case, case["kind"]
    if kind in ("infer", "train"):
        mac = sum(o * i for o, i in _layer_dims(c)) + 6 * c["freqs"]
        n = sum(o * i + o for o, i in _layer_dims(c))
        if kind == "infer":
            return {"bytes": 4 * n + 32 * c["n"], "flops": 2 * mac * c["n"]}
        return {"bytes": 4 * 8 * n + 32 * c["n"], "flops": 6 * mac * c["n"]}
    if kind == "freq":
        paths = c["pairs"] * c["mean_paths"]
        return {"bytes": paths * (8 * c["ports"] + 4) + 8 * c["pairs"] * c["ports"] * c["sc"],
                "flops": paths * c["sc"] * (8 * c["ports"] + 6)}
    T = 12 * c["n_side"] ** 2 + 2 if c["n_side"] else 14
    seg = 22 * math.log2(T) + 35
    n_tx = c.get("n_tx", 1)
    scene = 40 * T
    if kind == "links":
        pairs = n_tx * c["n_rx"]
        return {"bytes": scene + 8 * pairs * c["sc"], "flops": seg * (n_tx * c["rays"] * c["depth"] + pairs)}
    if kind == "labels":
        return {"bytes": scene + 32 * n_tx * c["n_rx"], "flops": seg * n_tx * (c["rays"] * c["depth"] + c["n_rx"])}
    if kind in ("coverage", "coverage_vjp"):
        return {"bytes": scene + (8 if kind == "coverage" else 4) * n_tx * c["nx"] * c["ny"],
                "flops": seg * n_tx * c["rays"] * (c["depth"] + 1)}
    if kind == "gradient":   # the stored paths replayed: H(f) of every pair, forward and backward
        ports = len(ANTENNAS[c["tx_ant"]].slants) * len(ANTENNAS[c["rx_ant"]].slants)
        return {"bytes": 3 * 8 * c["n_rx"] * ports * c["sc"], "flops": 3 * 8 * c["n_rx"] * ports * c["sc"]}
    if kind == "scattering":
        return {"bytes": scene + 4 * n_tx * c["n_rx"],
                "flops": n_tx * c["rays"] * seg * (1 + 0.5 * c["n_rx"])}
    # diffraction map: the Keller point of every (cell, wedge), about 60 operations
    return {"bytes": scene + 4 * n_tx * c["nx"] * c["ny"],
            "flops": 60 * n_tx * c["nx"] * c["ny"] * 12 * c["n_side"] ** 2}


# ------------------------------------------------------------------------ exact
def _exact_freq(c, seed):
    off, a, tau, freqs = _path_list(c, seed)
    pair = torch.as_tensor(np.repeat(np.arange(c["pairs"]), np.diff(off)), device="cuda")
    a = torch.as_tensor(a, device="cuda").to(torch.complex128)
    tau = torch.as_tensor(tau, device="cuda").double()
    f = torch.as_tensor(freqs, device="cuda")
    H = torch.zeros((c["pairs"], c["ports"], c["sc"]), dtype=torch.complex128, device="cuda")
    for s in range(0, len(tau), 2048):
        w = torch.exp(-2j * math.pi * torch.remainder(tau[s:s + 2048, None] * f[None], 1.0))
        for q in range(c["ports"]):
            H[:, q].index_add_(0, pair[s:s + 2048], a[s:s + 2048, q, None] * w)
    return torch.view_as_real(H).contiguous()


def _exact_forward(c, p, x):
    """(logit, scaled gain) of the network in 64 bits; p: the parameter tensors, x: float64 queries."""
    lo, hi = (torch.as_tensor(v, dtype=torch.float32, device="cuda").double() for v in BOX)
    B = p[-1].reshape(c["freqs"], 6)
    ang = 2.0 * math.pi * torch.remainder((2.0 * (x - lo) / (hi - lo) - 1.0) @ B.T, 1.0)
    h = torch.cat([torch.sin(ang), torch.cos(ang)], 1)
    for k, (o, i) in enumerate(_layer_dims(c)):
        h = h @ p[2 * k].reshape(o, i).T + p[2 * k + 1]
        if o > 2 or k < c["hidden"]:
            h = torch.relu(h)
    return h


def _split(c, p):
    sizes = [n for o, i in _layer_dims(c) for n in (o * i, o)] + [6 * c["freqs"]]
    return [v.clone() for v in p.double().split(sizes)]


def exact(case, seed):
    """In 64 bits: H(f) of a path list, the network's answers and its
    gradients. The traced cases have no such value within the time allowed
    (brute force over 5000 triangles takes minutes in numpy)."""
    c = case
    if c["kind"] == "freq":
        return _exact_freq(c, seed)
    if c["kind"] not in ("infer", "train"):
        return None
    p, x, t = _network(c, seed)
    p, x, t = _split(c, p), x.double(), t.double()
    if c["kind"] == "infer":
        out = [_exact_forward(c, p, x[s:s + (1 << 17)]) for s in range(0, len(x), 1 << 17)]
        y = torch.cat(out)
        return torch.stack([y[:, 0], 20.0 * y[:, 1] - 100.0], 1)
    for v in p[:-1]:
        v.requires_grad_(True)
    y = _exact_forward(c, p, x)
    has = t[:, 0]
    loss = (torch.nn.functional.binary_cross_entropy_with_logits(y[:, 0], has, reduction="none") +
            has * (y[:, 1] - (t[:, 1] + 100.0) / 20.0) ** 2).mean()
    loss.backward()
    grads = torch.cat([v.grad.reshape(-1) for v in p[:-1]] + [torch.zeros_like(p[-1])])
    return {"loss": loss.detach().reshape(1), "grads": grads}
