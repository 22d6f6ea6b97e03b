"""The work that this framework is used for, as cases that can be timed and whose outputs can be compared.

Kinds of case (sizes as in the repository's workloads, tests and benchmark):

* ``lattice``: one lattice of the fused LB freezing step: a chunk of steps, then the macroscopic fields
  (and, with ``diag``, the diagnostics that a freezing run logs);
* ``batch``: a parameter sweep of uneven droplets advanced together, then every instance's fields;
* ``jump``: the hand-over between the LB and the surrogate around the network: acceptance checks, network
  input, update of the fields, re-initialisation of the lattice and its first step;
* ``forward``: the surrogate network's forward pass on one lattice;
* ``train``: training steps of the network on mini-batches, and the gradients;
* ``layer``: one 3x3 convolution layer of the network: forward, data gradient, weight gradient.
"""
import math

import numpy as np
import torch

from paper_2511_09422_gb300 import cno, lbfreeze
from paper_2511_09422_gb300 import workloads as W

STORAGE = {"f32": (0, 0), "f16": (1, 0), "f16h32": (2, 0), "f32_d2q5": (0, 1)}  # (pop_storage, lattice_fl)
FIELDS = ("phi", "T", "fs", "C", "ux", "uy", "p")


def listed():
    return [
        # a film freezing on a cold wall (validation runs of thousands of steps): the smallest lattice, where the latency of a step counts
        dict(name="film_64x256", kind="lattice", setup="film", nx=64, ny=256, storage="f32", steps=20, diag=False),
        # the heated two-layer channel: no phase change, wall temperature varying along x
        dict(name="channel_512x256", kind="lattice", setup="channel", nx=512, ny=256, storage="f32", steps=20, diag=False),
        # a binary droplet on the way to full freezing, its diagnostics read after every chunk
        dict(name="droplet_512", kind="lattice", setup="droplet", nx=512, ny=512, storage="f32", steps=20, diag=True),
        # a liquid bridge between two wetting walls, an odd size, D2Q5 phase-field and solute sets
        dict(name="bridge_1037x771_d2q5", kind="lattice", setup="bridge", nx=1037, ny=771, storage="f32_d2q5", steps=10, diag=False),
        # the front toward an insoluble impurity with half-precision populations (FP32 enthalpy)
        dict(name="impurity_2048_f16h32", kind="lattice", setup="impurity", nx=2048, ny=2048, storage="f16h32", steps=10, diag=False),
        # the benchmark's lattice, the largest
        dict(name="impurity_4096", kind="lattice", setup="impurity", nx=4096, ny=4096, storage="f32", steps=4, diag=True),
        # a sweep over droplets of uneven sides, as for training data or a parameter study
        dict(name="sweep_64", kind="batch", instances=64, side_min=128, side_max=512, storage="f32", steps=10),
        # one surrogate jump's hand-over on a mid-sized lattice
        dict(name="jump_1024", kind="jump", nx=1024, ny=1024),
        # the network's prediction for that lattice
        dict(name="forward_1024", kind="forward", h=1024, w=1024),
        # training at the size the surrogate is trained at
        dict(name="train_16x256", kind="train", n=16, h=256, w=256, batches=3),
        # the full-resolution layer of a training batch, the network's most frequent one
        dict(name="layer_64to64_16x256", kind="layer", n=16, h=256, w=256, cin=64, cout=64),
        # a wide layer on a small ragged image
        dict(name="layer_256to128_2x50x168", kind="layer", n=2, h=50, w=168, cin=256, cout=128),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("lattice", "lattice", "lattice", "lattice", "batch", "jump", "forward", "train", "layer", "layer"))
    if kind == "lattice":
        return dict(kind=kind, setup=rng.choice(("film", "channel", "droplet", "bridge", "impurity")), nx=_log(rng, 48, 3000),
                    ny=_log(rng, 48, 3000), storage=rng.choice(("f32", "f32", "f16", "f16h32", "f32_d2q5")),
                    steps=rng.randint(4, 8), diag=rng.random() < 0.5)
    if kind == "batch":
        lo = rng.randint(64, 256)
        return dict(kind=kind, instances=_log(rng, 4, 64), side_min=lo, side_max=rng.randint(lo, 512),
                    storage=rng.choice(("f32", "f16h32")), steps=rng.randint(2, 20))
    if kind == "jump":
        return dict(kind=kind, nx=_log(rng, 96, 2048), ny=_log(rng, 96, 2048))
    if kind == "forward":  # widths whose coarser levels keep whole tiles: powers of two, or 1024 and more
        w = rng.choice((64, 128, 256, 512, 8 * rng.randint(128, 180)))
        return dict(kind=kind, h=8 * _log(rng, 4, 160), w=w)
    if kind == "train":
        return dict(kind=kind, n=rng.randint(1, 16), h=8 * rng.randint(4, 32), w=rng.choice((64, 128, 256)), batches=rng.randint(1, 3))
    return dict(kind=kind, n=rng.randint(1, 8), h=_log(rng, 8, 256), w=rng.choice((16, 32, 64, rng.randint(128, 300))),
                cin=64 * rng.choice((1, 2, 4)), cout=64 * rng.choice((1, 2, 3, 4)))


# ---- inputs -----------------------------------------------------------------------------------------------------------


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _lattice(setup, nx, ny, storage, seed):
    """Grid, parameters and FP32 device fields of one lattice; the seed moves the geometry a little and gives the noise."""
    rng = np.random.default_rng(seed)
    gen = _generator(seed)
    y, x = torch.meshgrid(torch.arange(ny, dtype=torch.float32, device="cuda"), torch.arange(nx, dtype=torch.float32, device="cuda"),
                          indexing="ij")

    def noise(lo):
        return torch.empty((ny, nx), dtype=torch.float32, device="cuda").uniform_(lo, 1.0, generator=gen)

    def tanh(d):
        return torch.tanh(2.0 * d / W.INTERFACE_WIDTH)

    jitter, c0, small = float(rng.uniform(-2.0, 2.0)), 0.05, min(nx, ny)
    if setup == "film":
        phi = tanh(0.5 * ny - 0.5 + jitter - y)
        p = W.gas_properties(W.base_params(rho_s=0.9, latent=10.0), 0.1)
        g = W.grid(nx, ny, T_bottom=-1.0)
        temp, conc = 1e-3 * noise(0.0), torch.zeros_like(phi)
    elif setup == "channel":
        h = ny // 2
        phi = tanh(h - 0.5 + jitter - y)
        p = W.base_params(mu_l=0.2, mu_s=0.2, mu_g=0.2, lam_l=0.2, lam_s=0.2, lam_g=0.2, latent=0.0, sigma0=2.5e-2,
                          sigma_T=-0.1 * 0.2 * 0.2 / (4.0 * h), T_ref=10.0, phase_change_on=0)
        g = W.grid(nx, ny, W.WALL_DIRICHLET_T, W.WALL_DIRICHLET_T, T_bottom=20.0, T_top=10.0, T_bottom_amp=4.0)
        temp, conc = 20.0 - 10.0 * (y + 0.5) / ny + 1e-3 * noise(-1.0), torch.zeros_like(phi)
    elif setup in ("droplet", "impurity"):
        if setup == "droplet":
            r = 0.2 * small + jitter
            d = r - torch.sqrt((x - 0.5 * nx) ** 2 + (y + 0.5) ** 2)
            rho_g, ratio = 0.1, 0.1
        else:
            r = 200.0 * small / 4096.0 + jitter + 4.0
            d = torch.sqrt((x - 0.5 * nx) ** 2 + (y - 0.25 * ny) ** 2) - r
            rho_g, ratio = 2.0, 1.0
        phi = tanh(d)
        p = W.gas_properties(W.base_params(rho_s=0.9, k_p=0.5, D_l=0.05, D_s=0.005, sigma0=0.01, latent=10.0, c_ref=c0),
                             rho_g, lam_ratio=ratio)
        p["sigma_T"], p["sigma_c"] = -10.0 * 0.1 * 0.3 / r, -10.0 * 0.1 * 0.05 / (c0 * r)
        g = W.grid(nx, ny, T_bottom=-1.0)
        temp = 1e-3 * noise(0.0)
        conc = c0 * (0.5 * (1.0 + phi)).clamp(0.0, 1.0) * (1.0 + 1e-3 * noise(-1.0))
    else:  # bridge
        phi = tanh(0.2 * nx + jitter - (x - 0.5 * (nx - 1)).abs())
        p = W.gas_properties(W.base_params(rho_s=0.9, latent=10.0, k_p=0.5, D_l=0.05, D_s=0.005, sigma0=0.01, sigma_T=-1e-3,
                                           sigma_c=-2e-2, c_ref=c0), 0.1)
        g = W.grid(nx, ny, W.WALL_DIRICHLET_T, W.WALL_DIRICHLET_T, T_bottom=-1.0, T_top=0.5, theta_bottom=60.0, theta_top=45.0)
        temp = 1e-3 * noise(0.0)
        conc = c0 * (phi > 0).float() * (1.0 + 1e-3 * noise(-1.0))
    p["pop_storage"], p["lattice_fl"] = STORAGE[storage]
    # a flow under way: one pair of divergence-free rolls between the walls, at rest on them
    k, a = 2.0 * math.pi / nx, 1e-3 * small / math.pi
    ux = a * math.pi / ny * torch.sin(k * x) * torch.sin(2.0 * math.pi * (y + 0.5) / ny)
    uy = -a * k * torch.cos(k * x) * torch.sin(math.pi * (y + 0.5) / ny) ** 2
    return g, p, dict(phi=phi, T=temp, C=conc.contiguous(), ux=ux, uy=uy)


def _sweep(case, seed):
    """Seeded droplets of uneven sides (the same sides for every seed): grids, parameters and host fields."""
    rng = np.random.default_rng(seed)
    sides = np.random.default_rng(20251109).integers(case["side_min"], case["side_max"] + 1, size=case["instances"])
    out = []
    for side in (int(v) for v in sides):
        g, p, f = _lattice("droplet", side, side, case["storage"], int(rng.integers(1 << 30)))
        p["latent"] = 1.0 / float(rng.uniform(0.05, 0.5))
        g["cos_theta_bottom"] = math.cos(math.radians(float(rng.uniform(60.0, 120.0))))
        out.append(dict(grid=g, params=p, fields={k: v.cpu().numpy() for k, v in f.items()}))
    return out


def _jump_inputs(case, seed):
    """Fields as the LB leaves them part-way through a freezing run, a prediction of the network, and its scales."""
    nx, ny = case["nx"], case["ny"]
    g, p, f = _lattice("impurity", nx, ny, "f32", seed)
    gen = _generator(seed + 1)

    def noise(a):
        return a * torch.randn((ny, nx), device="cuda", generator=gen)

    chi = (0.5 * (1.0 + f["phi"])).clamp(0.0, 1.0)
    rows = torch.arange(ny, dtype=torch.float32, device="cuda").reshape(ny, 1)
    f["fs"] = (chi * torch.sigmoid(0.1 * ny - rows)).contiguous()
    f["T"] = (-torch.sigmoid(0.1 * ny - rows) + f["T"]).contiguous()
    f["ux"], f["uy"], f["p"] = f["ux"] + noise(1e-5), f["uy"] + noise(1e-5), noise(1e-5)
    pred = torch.randn((1, ny, nx, cno.NF), device="cuda", generator=gen)
    offset = np.array([0.9, -0.1, 0.1, 0.045, 0.0, 0.0, 0.0], np.float32)
    inv_scale = np.array([2.0, 4.0, 4.0, 50.0, 5e3, 5e3, 5e4], np.float32)
    scale = np.array([1e-3, 1e-3, 1e-3, 1e-4, 0.0, 0.0, 0.0], np.float32)
    hcoef = tuple(float(np.float32(v)) for v in (p["rho_l"] * p["cp_l"], p["rho_s"] * p["cp_s"], p["rho_g"] * p["cp_g"],
                                                   p["rho_l"] * p["latent"]))
    inf = float("inf")
    return dict(g=g, p=p, cur=f, pred=pred, offset=offset, inv_scale=inv_scale, scale=scale, hcoef=hcoef,
                lo=[-1.0, -1.0, 0.0, 0.0, -inf, -inf, -inf], hi=[1.0, 1.0, 1.0, inf, inf, inf, inf])


def _network(seed):
    """He-normal weights, small biases, in the order of the flat parameter vector."""
    rng = np.random.default_rng(seed)
    out = []
    for ci, co in cno.layer_shapes():
        out += [(rng.standard_normal(co * 9 * ci, dtype=np.float32) * np.float32(math.sqrt(2.0 / (9 * ci)))),
                0.05 * rng.standard_normal(co, dtype=np.float32)]
    return np.concatenate(out)


def _images(n, h, w, seed):
    """Network input: seven normalised fields, zero in the other channels."""
    gen = _generator(seed)
    x = torch.zeros((n, h, w, cno.CIN), dtype=torch.bfloat16, device="cuda")
    x[..., :cno.NF] = torch.randn((n, h, w, cno.NF), device="cuda", generator=gen).to(torch.bfloat16)
    return x, torch.randn((n, h, w, cno.NF), device="cuda", generator=gen)


def _layer(case, seed):
    gen = _generator(seed)
    n, h, w, ci, co = (case[k] for k in ("n", "h", "w", "cin", "cout"))

    def randn(*shape):
        return torch.randn(shape, device="cuda", generator=gen)

    return dict(x=randn(n, h, w, ci).to(torch.bfloat16), dz=randn(n, h, w, co).to(torch.bfloat16),
                w32=randn(co, 9, ci) / math.sqrt(9 * ci), b=0.1 * randn(co))


# ---- the calls ----------------------------------------------------------------------------------------------------------


def _outputs(nx, ny):
    return {k: torch.empty((ny, nx), dtype=torch.float32, device="cuda") for k in FIELDS}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        g, p, f = _lattice(case["setup"], case["nx"], case["ny"], case["storage"], seed)
        return dict(kind=kind, steps=case["steps"], diag=case["diag"], solver=lbfreeze.Solver(g, p, f), out=_outputs(case["nx"], case["ny"]))
    if kind == "batch":
        batch = lbfreeze.Batch(_sweep(case, seed))
        out = torch.empty(7 * batch.cells, dtype=torch.float32, device="cuda")
        views, at = [], 0
        for nx, ny in batch.shapes:
            views.append({k: out[at + i * nx * ny:at + (i + 1) * nx * ny].view(ny, nx) for i, k in enumerate(FIELDS)})
            at += 7 * nx * ny
        return dict(kind=kind, steps=case["steps"], batch=batch, inst=[batch.instance(i) for i in range(batch.n)], views=views, out=out)
    if kind == "jump":
        s = _jump_inputs(case, seed)
        nx, ny = case["nx"], case["ny"]
        return dict(s, kind=kind, solver=lbfreeze.Solver(s["g"], s["p"], {k: s["cur"][k] for k in ("phi", "T", "C")}), new=_outputs(nx, ny),
                    next=_outputs(nx, ny), x=torch.empty((1, ny, nx, cno.CIN), dtype=torch.bfloat16, device="cuda"))
    if kind in ("forward", "train"):
        net = cno.Net()
        net.set_params(_network(seed))
        n = case.get("n", 1)
        batches = [_images(n, case["h"], case["w"], seed + 1000 * k) for k in range(case.get("batches", 1))]
        return dict(kind=kind, net=net, batches=batches, out=torch.empty((n, case["h"], case["w"], cno.NF), device="cuda"))
    s = _layer(case, seed)
    s["wf"], s["wd"] = cno.weights_to_bf16(s["w32"])
    return dict(s, kind=kind)


def run(s):
    kind = s["kind"]
    if kind == "lattice":
        s["solver"].step(s["steps"])
        out = dict(s["solver"].fields(out=s["out"]))
        if s["diag"]:  # as a run logs them, in single precision
            out["diag"] = s["solver"].reduce().astype(np.float32)
        return out
    if kind == "batch":
        s["batch"].step(s["steps"])
        for inst, out in zip(s["inst"], s["views"]):
            inst.fields(out=out)
        return s["out"]
    if kind == "jump":
        cur, new = s["cur"], s["new"]
        before = cno.field_checks(cur["phi"], cur["fs"], cur["T"], s["hcoef"])
        cno.pack_fields([cur[k] for k in FIELDS], s["offset"], s["inv_scale"], out=s["x"])
        cno.apply_update([cur[k] for k in FIELDS], [new[k] for k in FIELDS], s["pred"], s["scale"], 0.999, s["lo"], s["hi"])
        after = cno.field_checks(new["phi"], new["fs"], new["T"], s["hcoef"])
        s["solver"].set_fields(new)
        s["solver"].step(1)
        s["solver"].fields(out=s["next"])
        return dict(before=list(before), after=list(after), x=s["x"], new=new, next=s["next"])
    if kind == "forward":
        return s["net"].forward(s["batches"][0][0], out=s["out"])
    if kind == "train":
        # learning rate 0, the first step of a warm-up: all of a training step, and the same weights for the next pass
        last = len(s["batches"]) - 1
        for k, (x, t) in enumerate(s["batches"]):
            loss = s["net"].train_step(x, t, 0.0, update=True, want_loss=k == last)
        return dict(loss=np.float32(loss), grads=s["net"].grads())
    y = cno.conv3x3_forward(s["x"], s["wf"], s["b"], True)
    dx = cno.conv3x3_dgrad(s["dz"], s["wd"], s["x"])
    dw, db = cno.conv3x3_wgrad(s["dz"], s["x"])
    return dict(y=y, dx=dx, dw=dw, db=db)


# ---- what a pass cannot do without ---------------------------------------------------------------------------------------


def _update_bytes(storage):
    return {"f32": 352.0, "f16": 208.0, "f16h32": 244.0, "f32_d2q5": 288.0}[storage]


def work(case):
    kind = case["kind"]
    if kind == "lattice":
        cells, pops = case["nx"] * case["ny"], (_update_bytes(case["storage"]) - 64.0) / 2.0
        read = pops + 32.0 + 28.0  # the fields: the state read, seven planes written
        diag = (0.75 * pops + 16.0) if case["diag"] else 0.0
        return dict(bytes=cells * (case["steps"] * _update_bytes(case["storage"]) + read + diag), flops=600.0 * cells * case["steps"])
    if kind == "batch":
        mid = (case["side_min"] + case["side_max"]) / 2.0
        cells = case["instances"] * (mid ** 2 + (case["side_max"] - case["side_min"]) ** 2 / 12.0)
        b = _update_bytes(case["storage"])
        return dict(bytes=cells * (case["steps"] * b + (b - 64.0) / 2.0 + 60.0), flops=600.0 * cells * case["steps"])
    if kind == "jump":
        # two checks of 12 B, the input 28 -> 128 B, the update 28 + 28 -> 28 B, the state from 28 B (176 B), one step, the fields
        return dict(bytes=case["nx"] * case["ny"] * (2 * 12.0 + 156.0 + 84.0 + 28.0 + 176.0 + 352.0 + 204.0), flops=800.0 * case["nx"] * case["ny"])
    if kind in ("forward", "train"):
        n, h, w = case.get("n", 1), case["h"], case["w"]
        passes = 1.0 if kind == "forward" else 3.0 * case["batches"]
        flops = passes * cno.forward_flops(h, w, n)
        pix = n * h * w
        params = sum(co * (9 * ci + 1) for ci, co in cno.layer_shapes())
        b = pix * (2 * cno.CIN + 4 * cno.NF) * (1 if kind == "forward" else case["batches"])
        return dict(bytes=float(b + params * (2 if kind == "forward" else 28 * case["batches"])), flops=float(flops))
    pix, ci, co = case["n"] * case["h"] * case["w"], case["cin"], case["cout"]
    return dict(bytes=float(pix * (2 * (ci + co) * 2 + 2 * (ci + co) + 2 * ci) + 9 * ci * co * 8), flops=3.0 * 18.0 * pix * ci * co)


# ---- the same in 64 bits ----------------------------------------------------------------------------------------------------

_CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
_CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
_OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
_W9 = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
_W5 = (1 / 3,) + (1 / 6,) * 4 + (0.0,) * 4


class _Reference:
    """The method's step in FP64 torch operations: collide, then stream, populations in post-streaming form."""

    def __init__(self, g, p, f, handed_back=False):
        self.g, self.p = g, p
        f = {k: v.double() for k, v in f.items()}
        self.wfl = _W5 if p.get("lattice_fl") else _W9
        self.rr = p["rho_l"] * 2.0 * p["cp_s"] * p["cp_l"] / (p["cp_s"] + p["cp_l"])
        self.rcp = [p["rho_" + k] * p["cp_" + k] for k in "lsg"]
        phi, T, C = f["phi"], f["T"], f["C"]
        zero = torch.zeros_like(phi)
        ux, uy, pr = f.get("ux", zero), f.get("uy", zero), f.get("p", zero)
        chi = (0.5 * (1.0 + phi)).clamp(0.0, 1.0)
        Al, As = chi * self.rcp[0] + (1 - chi) * self.rcp[2], chi * self.rcp[1] + (1 - chi) * self.rcp[2]
        if not p["phase_change_on"]:
            fs, rhoH = zero, Al * T
        elif "fs" in f:
            fs = torch.minimum(f["fs"].clamp(min=0.0), chi)
            rhoH = T * (fs * self.rcp[1] + (chi - fs) * self.rcp[0] + (1 - chi) * self.rcp[2]) + p["rho_l"] * p["latent"] * (chi - fs)
        else:  # T_sol = T_liq in every case here
            fs = torch.where(T < p["T_sol"], chi, zero)
            rhoH = torch.where(T < p["T_sol"], As * T, Al * T + chi * p["rho_l"] * p["latent"])
        self.lag = dict(fs=fs, Q=zero, phi=phi, C=C, ux=ux, uy=uy, p=pr, S=zero)
        eq = self._equilibria(phi, C, rhoH, T, pr, ux, uy, self._zeta(phi, fs, "rho"), self._rcp(phi, fs))
        self.pop = {s: torch.stack(eq[s]) for s in "fghl"}
        if handed_back and p["divu_mode"]:
            self.pop["f"][0] -= 0.5 * phi * (self._grad(ux, "u")[0] + self._grad(uy, "u")[1])

    def _zeta(self, phi, fs, name):
        zl, zs, zg = (self.p["%s_%s" % (name, k)] for k in "lsg")
        return 0.5 * phi * (zl - zg) + fs * (zs - zl) + 0.5 * (zl + zg)

    def _rcp(self, phi, fs):
        zl, zs, zg = self.rcp
        return 0.5 * phi * (zl - zg) + fs * (zs - zl) + 0.5 * (zl + zg)

    def _wall_T(self, bottom):
        g = self.g
        if not bottom:
            return g["T_top"]
        x = torch.arange(g["nx"], dtype=torch.float64, device="cuda")
        return g["T_bottom"] + g["T_bottom_amp"] * torch.cos(2.0 * math.pi * g["T_bottom_modes"] * x / g["nx"])

    def _padded(self, v, kind):
        g, lo, hi = self.g, v[0], v[-1]
        if kind == "u":
            lo, hi = -lo, -hi
        elif kind == "T":
            lo = 2.0 * self._wall_T(True) - lo if g["bc_bottom"] == W.WALL_DIRICHLET_T else lo
            hi = 2.0 * self._wall_T(False) - hi if g["bc_top"] == W.WALL_DIRICHLET_T else hi
        elif kind == "phi":
            k = 1.0 / (math.sqrt(2.0) * self.p["eps"])
            lo, hi = lo + g["cos_theta_bottom"] * k * (1 - lo * lo), hi + g["cos_theta_top"] * k * (1 - hi * hi)
        return torch.cat([lo[None], v, hi[None]])

    def _grad(self, v, kind="mirror", laplacian=False):
        q, ny = self._padded(v, kind), v.shape[0]
        gx, gy, lap = torch.zeros_like(v), torch.zeros_like(v), torch.zeros_like(v)
        for i in range(1, 9):
            d = torch.roll(q[1 + _CY[i]:1 + _CY[i] + ny], -_CX[i], 1) - v
            gx += 3.0 * _W9[i] * _CX[i] * d
            gy += 3.0 * _W9[i] * _CY[i] * d
            lap += 6.0 * _W9[i] * d
        return (gx, gy, lap) if laplacian else (gx, gy)

    def _equilibria(self, phi, C, rhoH, T, pr, ux, uy, rho, rhocp):
        uu, rr = ux * ux + uy * uy, self.rr
        out = dict(f=[], g=[], h=[], l=[])
        for i in range(9):
            cu = _CX[i] * ux + _CY[i] * uy
            out["f"].append(self.wfl[i] * phi * (1 + 3 * cu))
            out["l"].append(self.wfl[i] * C * (1 + 3 * cu))
            out["g"].append(3 * pr * (_W9[i] - (i == 0)) + rho * _W9[i] * (3 * cu + 4.5 * cu * cu - 1.5 * uu))
            h = _W9[i] * (rr * T + rhocp * T * (3 * cu + 4.5 * cu * cu - 1.5 * uu))
            out["h"].append(h + rhoH - rr * T if i == 0 else h)
        return out

    def _local(self):
        p, lag = self.p, self.lag
        sf, C = self.pop["f"].sum(0), self.pop["l"].sum(0)
        e = self.pop["h"].sum(0) + 0.5 * lag["Q"]
        div, phi = None, None
        if p["divu_mode"]:
            div = self._grad(lag["ux"], "u")[0] + self._grad(lag["uy"], "u")[1]
            phi = sf / (1 - 0.5 * div)
        chi = (0.5 * (1 + (sf if phi is None else phi))).clamp(0.0, 1.0)
        Al, As = chi * self.rcp[0] + (1 - chi) * self.rcp[2], chi * self.rcp[1] + (1 - chi) * self.rcp[2]
        zero = torch.zeros_like(e)
        if p["phase_change_on"]:
            lat = chi * p["rho_l"] * p["latent"]
            Es, El = As * p["T_sol"], Al * p["T_liq"] + lat
            r = torch.where(El - Es < 1e-14 * e.abs().clamp(min=1.0), torch.ones_like(e), (e - Es) / (El - Es).clamp(min=1e-300))
            fs = torch.where(e < Es, chi, torch.where(e > El, zero, chi * (1 - r)))
            T = torch.where(e < Es, e / As, torch.where(e > El, p["T_liq"] + (e - El) / Al, p["T_sol"] + r * (p["T_liq"] - p["T_sol"])))
            mdot = (1 - p["rho_s"] / p["rho_l"]) * (fs - lag["fs"])
        else:
            fs, T, mdot = zero, e / Al, zero
        if div is None:
            div = mdot
            phi = sf / (1 - 0.5 * div)
        return phi, T, fs, C, e, mdot, div

    def _dynamics(self):
        p, lag, pop = self.p, self.lag, self.pop
        phi, T, fs, C, e, mdot, div = self._local()
        m = dict(phi=phi, T=T, fs=fs, C=C, e=e, div=div)
        gpx, gpy, lap = self._grad(phi, "phi", True)
        gTx, gTy = self._grad(T, "T")
        gCx, gCy = self._grad(C)
        gfx, gfy = self._grad(fs)
        rho, mu = self._zeta(phi, fs, "rho"), self._zeta(phi, fs, "mu")
        grx, gry = (0.5 * (p["rho_l"] - p["rho_g"]) * a + (p["rho_s"] - p["rho_l"]) * b for a, b in ((gpx, gfx), (gpy, gfy)))
        g2 = gpx * gpx + gpy * gpy
        inv = 1 / torch.sqrt(g2 + 1e-6)
        m["nx"], m["ny"] = gpx * inv, gpy * inv
        chem = (phi ** 3 - phi) / p["eps"] ** 2 - lap
        sigma = p["sigma0"] + p["sigma_T"] * (T - p["T_ref"]) + p["sigma_c"] * (C - p["c_ref"])
        sx, sy = p["sigma_T"] * gTx + p["sigma_c"] * gCx, p["sigma_T"] * gTy + p["sigma_c"] * gCy
        al, dot = 3 * math.sqrt(2.0) * p["eps"] / 4, sx * gpx + sy * gpy
        mod = (1 - fs) if p["fs_modulated_st"] else 1.0
        Fx = mod * al * (g2 * sx - dot * gpx + sigma * chem * gpx) + rho * p["gx"]
        Fy = mod * al * (g2 * sy - dot * gpy + sigma * chem * gpy) + rho * p["gy"]
        jx = sum(_CX[i] * pop["g"][i] for i in range(1, 9))
        jy = sum(_CY[i] * pop["g"][i] for i in range(1, 9))
        sx, sy = (jx + 0.5 * Fx) / rho, (jy + 0.5 * Fy) / rho
        m["rfx"], m["rfy"] = -rho * fs * sx, -rho * fs * sy
        ux, uy = sx * (1 - 0.5 * fs), sy * (1 - 0.5 * fs)
        S = rho * mdot + ux * grx + uy * gry
        gPx, gPy = self._grad(lag["p"])
        gSx, gSy = self._grad(lag["S"])
        Ftx, Fty = Fx - gPx + (grx + gSx) / 3, Fy - gPy + (gry + gSy) / 3
        uu, uF, tau = ux * ux + uy * uy, ux * Ftx + uy * Fty, 0.5 + 3 * mu / rho
        pr = 0.6 * (pop["g"][1:].sum(0) + 0.5 * S + tau * _W9[0] * (S - 3 * uF) - rho * _W9[0] * 1.5 * uu)
        m.update(ux=ux, uy=uy, p=pr, S=S, Fx=Fx, Fy=Fy, Ftx=Ftx, Fty=Fty, uF=uF, tau=tau, rho=rho, gfx=gfx, gfy=gfy)
        return m

    def fields(self):
        m = self._dynamics()
        return {k: m[k] for k in FIELDS}

    def diag(self, V0):
        phi, T, fs, C, e, _, _ = self._local()
        chi = (0.5 * (1 + phi)).clamp(0.0, 1.0)
        s = [float(v.sum()) for v in (phi, e, C, fs, chi, fs[:, self.g["nx"] // 2])]
        return torch.tensor(s + [s[3] / V0, s[4] / V0], dtype=torch.float64)

    def step(self):
        p, lag, pop, m = self.p, self.lag, self.pop, self._dynamics()
        phi, T, fs, C, ux, uy, S, rho = (m[k] for k in ("phi", "T", "fs", "C", "ux", "uy", "S", "rho"))
        rhocp, s2e = self._rcp(phi, fs), math.sqrt(2.0) * p["eps"]
        Q = rhocp * T * m["div"]
        eq = self._equilibria(phi, C, m["e"], T, m["p"], ux, uy, rho, rhocp)
        kf = (1 - phi * phi) / (3 * s2e)
        ax, ay = phi * ux - lag["phi"] * lag["ux"] + kf * m["nx"], phi * uy - lag["phi"] * lag["uy"] + kf * m["ny"]
        keff = 1 - fs * (1 - p["k_p"])
        Rx, Ry = ((1 - phi) * C * n / s2e + (p["k_p"] - 1) * C * gf / keff for n, gf in ((m["nx"], m["gfx"]), (m["ny"], m["gfy"])))
        bx, by = C * ux - lag["C"] * lag["ux"] + Rx / 3, C * uy - lag["C"] * lag["uy"] + Ry / 3
        om_f, om_g = 1 / (0.5 + 3 * p["mobility"]), 1 / m["tau"]
        om_l = 1 / (0.5 + 3 * (fs * p["k_p"] * p["D_s"] + (1 - fs) * p["D_l"]) / keff)
        om_a = 1 / (0.5 + 3 * self._zeta(phi, fs, "lam") / self.rr)
        om_s = 2 - om_a
        new = {}
        for s in "fgl":
            out = []
            for i in range(9):
                cx, cy = _CX[i], _CY[i]
                if s == "f":
                    src = (1 - 0.5 * om_f) * self.wfl[i] * (3 * (cx * ax + cy * ay) + phi * m["div"])
                    om = om_f
                elif s == "g":
                    cu, cF = cx * ux + cy * uy, cx * m["Ftx"] + cy * m["Fty"]
                    src = (1 - 0.5 * om_g) * _W9[i] * (S + 3 * (cx * (m["Fx"] + m["rfx"]) + cy * (m["Fy"] + m["rfy"])) + 9 * cu * cF - 3 * m["uF"])
                    om = om_g
                else:
                    src = (1 - 0.5 * om_l) * self.wfl[i] * 3 * (cx * bx + cy * by)
                    om = om_l
                out.append(pop[s][i] - (pop[s][i] - eq[s][i]) * om + src)
            new[s] = out
        h, he = pop["h"], eq["h"]
        new["h"] = []
        for i in range(9):
            a, b = 0.5 * (h[i] + h[_OPP[i]]), 0.5 * (h[i] - h[_OPP[i]])
            ae, be = 0.5 * (he[i] + he[_OPP[i]]), 0.5 * (he[i] - he[_OPP[i]])
            if i == 0:
                ae, be = he[0], torch.zeros_like(b)
            new["h"].append(h[i] - om_s * (a - ae) - om_a * (b - be) + (1 - 0.5 * om_s) * _W9[i] * Q)
        for s in "fghl":
            for i in range(9):
                d = torch.roll(new[s][i], (_CY[i], _CX[i]), (0, 1))
                if _CY[i]:  # the row next to a wall, from the wall
                    row = 0 if _CY[i] > 0 else -1
                    back = new[s][_OPP[i]][row]
                    if s == "h" and self.g["bc_bottom" if row == 0 else "bc_top"] == W.WALL_DIRICHLET_T:
                        back = 2 * _W9[i] * self.rr * self._wall_T(row == 0) - back
                    d[row] = back
                pop[s][i] = d
            new[s] = None
        self.lag = dict(fs=fs, Q=Q, phi=phi, C=C, ux=ux, uy=uy, p=m["p"], S=S)


def _lattice_exact(g, p, f, steps, diag):
    r = _Reference(g, p, f)
    V0 = float((0.5 * (1 + f["phi"].double())).clamp(0.0, 1.0).sum())
    for _ in range(steps):
        r.step()
    out = r.fields()
    if diag:
        out["diag"] = r.diag(V0)
    return out


def _checks(F, hc):
    """The acceptance checks of a state."""
    phi, fs, T = (F[k].double() for k in ("phi", "fs", "T"))
    gx = 0.5 * (torch.roll(phi, -1, 1) - torch.roll(phi, 1, 1))
    gy = torch.empty_like(phi)
    gy[1:-1], gy[0], gy[-1] = 0.5 * (phi[2:] - phi[:-2]), phi[1] - phi[0], phi[-1] - phi[-2]
    chi = (0.5 * (1 + phi)).clamp(0.0, 1.0)
    s = torch.minimum(fs.clamp(min=0.0), chi)
    cl, cs, cg, lat = hc
    H = T * (s * cs + (chi - s) * cl + (1 - chi) * cg) + lat * (chi - s)
    v = (phi.sum(), chi.sum(), fs.sum(), (1 - phi * phi).sum(), torch.sqrt(gx * gx + gy * gy).sum(), T.min(), T.max(), H.sum())
    return [float(x) for x in v]


def _conv(x, w, b=None):
    """3x3 convolution of NCHW x with weights [o][9][i]."""
    o, _, i = w.shape
    return torch.nn.functional.conv2d(x, w.reshape(o, 3, 3, i).permute(0, 3, 1, 2), b, padding=1)


def _lrelu(z):
    return torch.where(z > 0, z, z / 16)


def _net_exact(flat, x):
    """The network in 64 bits: weights as the tensor cores take them, no rounding of activations."""
    par, at = [], 0
    for ci, co in cno.layer_shapes():
        w = flat[at:at + co * 9 * ci].reshape(co, 9, ci)
        par.append((w, flat[at + co * 9 * ci:at + co * (9 * ci + 1)]))
        at += co * (9 * ci + 1)
    pool, up = torch.nn.functional.avg_pool2d, lambda v: v.repeat_interleave(2, 2).repeat_interleave(2, 3)  # noqa: E731

    def layer(k, v, act=True):
        z = _conv(v, *par[k])
        return _lrelu(z) if act else z

    e0 = layer(1, layer(0, x))
    e1 = layer(3, layer(2, pool(e0, 2)))
    e2 = layer(5, layer(4, pool(e1, 2)))
    d = layer(7, layer(6, pool(e2, 2)))
    d = layer(8, up(d) + e2)
    d = layer(9, up(d) + e1)
    d = layer(10, up(d) + e0)
    return layer(11, d, False)[:, :cno.NF]


def _flat64(seed):
    """The flat parameters in 64 bits, weights rounded to bf16 and biases as they are."""
    flat, at = torch.from_numpy(_network(seed)).cuda(), 0
    out = flat.double()
    for ci, co in cno.layer_shapes():
        out[at:at + co * 9 * ci] = flat[at:at + co * 9 * ci].to(torch.bfloat16).double()
        at += co * (9 * ci + 1)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        return _lattice_exact(*_lattice(case["setup"], case["nx"], case["ny"], case["storage"], seed), case["steps"], case["diag"])
    if kind == "batch":
        out = []
        for w in _sweep(case, seed):
            f = {k: torch.from_numpy(v).cuda() for k, v in w["fields"].items()}
            r = _lattice_exact(w["grid"], w["params"], f, case["steps"], False)
            out += [r[k].reshape(-1) for k in FIELDS]
        return torch.cat(out)
    if kind == "jump":
        s = _jump_inputs(case, seed)
        cur = {k: v.double() for k, v in s["cur"].items()}
        new = {}
        for i, k in enumerate(FIELDS):
            sc = float(s["scale"][i])
            v = (cur[k] + sc * s["pred"][0, ..., i].double()).clamp(s["lo"][i], s["hi"][i])
            new[k] = cur[k] if sc == 0 else torch.where(cur[k].abs() >= float(np.float32(0.999)), cur[k], v) if k == "phi" else v
        x = torch.zeros((1, case["ny"], case["nx"], cno.CIN), dtype=torch.float64, device="cuda")
        for i, k in enumerate(FIELDS):
            x[0, ..., i] = (cur[k] - float(s["offset"][i])) * float(s["inv_scale"][i])
        r = _Reference(s["g"], s["p"], new, handed_back=True)
        r.step()
        return dict(before=_checks(cur, s["hcoef"]), after=None, x=x, new=new, next=r.fields())
    if kind == "forward":
        x = _images(1, case["h"], case["w"], seed)[0].double().permute(0, 3, 1, 2)
        return _net_exact(_flat64(seed), x).permute(0, 2, 3, 1).contiguous()
    if kind == "train":
        k = case["batches"] - 1
        x, t = _images(case["n"], case["h"], case["w"], seed + 1000 * k)
        flat = _flat64(seed).requires_grad_()
        loss, pix = 0.0, case["n"] * case["h"] * case["w"]
        for i in range(case["n"]):  # image by image, to bound the memory
            d = _net_exact(flat, x[i:i + 1].double().permute(0, 3, 1, 2)).permute(0, 2, 3, 1) - t[i:i + 1].double()
            part = (d * d).sum() / (pix * cno.NF)
            part.backward()
            loss += float(part)
        return dict(loss=loss, grads=flat.grad)
    s = _layer(case, seed)
    x, dz = (s[k].double().permute(0, 3, 1, 2) for k in ("x", "dz"))
    w = s["w32"].to(torch.bfloat16).double().requires_grad_()
    xg = x.clone().requires_grad_()
    z = _conv(xg, w)
    dx, dw = torch.autograd.grad(z, (xg, w), dz)
    y = _lrelu(z.detach() + s["b"].double().reshape(1, -1, 1, 1))
    dx = dx * torch.where(x > 0, 1.0, 1 / 16)
    return dict(y=y.permute(0, 2, 3, 1), dx=dx.permute(0, 2, 3, 1), dw=dw, db=dz.sum((0, 2, 3)))
