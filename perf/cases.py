"""The work this library does for its users, as cases that can be timed and checked.

A case is one of four ways a program uses the library:

* ``step``: one time step between the caller's own device buffers (lbm_step_noalloc), as programs
  do that own the populations or record the step into a graph of their own;
* ``solve``: one resonator solve from rest (create, step, read the force history, destroy);
* ``batch``: a sweep of instances of uneven sizes advanced together (lbm_batch_*);
* ``serve``: a burst of solve requests of both lattices to a running server (lbm_server_*).

The seed draws what a user varies between runs of one shape: the drive amplitude, the frequency
(within a few per cent of the case's), where the obstacles of a ``blocks`` geometry stand, and for
``step`` the flow it starts from.

A run's outputs are only as exact as its populations, so a solve hands its force history (and its
state, where the case reads it) back in the populations' storage type: FP64, FP32, FP16 or BF16.
The force is given per unit drive amplitude, F / u0, which keeps it in the range of every type.
``step`` returns the buffers that the library wrote.
"""
import math

import numpy as np
import torch

from paper_0904_4504_gb300 import lbm as L

STORAGE = {"f64": L.LBM_STORE_F64, "f32": L.LBM_STORE_F32, "bf16": L.LBM_STORE_BF16, "f16": L.LBM_STORE_F16}
DTYPE = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
GEOMETRY = {"plate": L.LBM_GEOM_PLATE, "beam": L.LBM_GEOM_BEAM, "blocks": L.LBM_GEOM_MASK}
DRIVE = {"wall": L.LBM_DRIVE_WALL, "body": L.LBM_DRIVE_BODYFORCE}
COLLISION = {"bgk": L.LBM_COLL_BGK, "reg": L.LBM_COLL_REGULARIZED}
WALLS = {"bounce": L.LBM_SCHEME_BOUNCEBACK, "diffuse": L.LBM_SCHEME_DIFFUSE}
LAYOUT = {"two": L.LBM_LAYOUT_AB, "inplace": L.LBM_LAYOUT_AA}
DEVICE = "cuda"


# ------------------------------------------------------------------------------------------------
# cases
# ------------------------------------------------------------------------------------------------

def _one(kind, lattice, nx, ny, geometry, storage, steps, *, lx=0, ly=0, drive="body", collision="reg", walls="bounce",
         layout="two", tau_omega=1.0, state=False):
    return {"kind": kind, "lattice": lattice, "nx": nx, "ny": ny, "geometry": geometry, "lx": lx, "ly": ly,
            "drive": drive, "collision": collision, "storage": storage, "walls": walls, "layout": layout,
            "tau_omega": tau_omega, "steps": steps, "state": state}


def _many(kind, lattice, storage, count, low, high, mix, steps, *, mode="streams", tau_omega=1.0):
    return {"kind": kind, "lattice": lattice, "storage": storage, "count": count, "low": low, "high": high, "mix": mix,
            "steps": steps, "mode": mode, "tau_omega": tau_omega}


def listed():
    cases = {
        # the smallest call: one step of the thickness-shear plate in the caller's buffers
        "step-plate-q9-f64-4x256": _one("step", 9, 4, 256, "plate", "f64", 1, drive="wall", collision="bgk", tau_omega=0.1),
        # one step of a caller's own loop over a mid-size section of odd sides in mixed precision
        "step-beam-q37-f16-1003x517": _one("step", 37, 1003, 517, "beam", "f16", 1, lx=32, ly=64),
        # the plate workload as configured: FP64, some 20 drive periods, field read back at the end
        "solve-plate-q9-f64-4x256": _one("solve", 9, 4, 256, "plate", "f64", 378, drive="wall", collision="bgk",
                                         tau_omega=0.1, state=True),
        # the sweep's smallest section, two periods: every array fits the caches, steps are short
        "solve-beam-q37-f32-256": _one("solve", 37, 256, 256, "beam", "f32", 256, lx=32, ly=32),
        # the beam the throughput figures are quoted on, two periods
        "solve-beam-q37-f32-1024": _one("solve", 37, 1024, 1024, "beam", "f32", 256, lx=32, ly=32),
        # the precision study's mixed-precision run on its full box, one period
        "solve-beam-q37-f16-2048": _one("solve", 37, 2048, 2048, "beam", "f16", 128, lx=32, ly=32, tau_omega=0.1),
        # the FP64 run that the other precisions are judged by
        "solve-beam-q37-f64-512": _one("solve", 37, 512, 512, "beam", "f64", 128, lx=32, ly=32, tau_omega=0.1),
        # the quartz plate of the quality-factor sweep with slip (diffuse walls) on its long narrow box
        "solve-plate-q37-f32-diffuse-32x4096": _one("solve", 37, 32, 4096, "plate", "f32", 256, drive="wall",
                                                    walls="diffuse", tau_omega=0.3),
        # a box of odd sides whose user needs the memory: one buffer, updated in place
        "solve-beam-q37-f32-inplace-1001x777": _one("solve", 37, 1001, 777, "beam", "f32", 128, lx=21, ly=210,
                                                    drive="wall", layout="inplace"),
        # part of the frequency and aspect-ratio sweep in mixed precision
        "batch-sweep-q37-f16": _many("batch", 37, "f16", 16, 256, 1024, 20090424, 256),
        # the same in FP32 as one persistent launch
        "batch-sweep-q37-f32-persistent": _many("batch", 37, "f32", 12, 256, 1024, 20090425, 128, mode="persistent"),
        # a burst of mixed requests (both lattices, plates and beams) to a server
        "serve-burst-f16": _many("serve", 0, "f16", 16, 128, 1024, 4504, 256),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def _log_int(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    kind = rng.choice(["step", "solve", "solve", "solve", "batch", "serve"])
    lattice = rng.choice([37, 37, 9])
    tau_omega = round(math.exp(rng.uniform(math.log(0.03), math.log(10.0))), 3)
    if kind in ("batch", "serve"):
        low = _log_int(rng, 96, 400)
        return _many(kind, lattice if kind == "batch" else 0, rng.choice(["f16", "f16", "f32", "bf16"]),
                     rng.randint(4, 14), low, rng.randint(low, 900), rng.randint(1, 1 << 30), 2 * rng.randint(64, 110),
                     mode=rng.choice(["streams", "persistent"]), tau_omega=tau_omega)
    geometry = rng.choice(["plate", "beam", "beam", "blocks"])
    walls = "diffuse" if kind == "solve" and rng.random() < 0.2 else "bounce"
    layout = "inplace" if kind == "solve" and walls == "bounce" and rng.random() < 0.2 else "two"
    storage = rng.choice(["f32", "f32", "f16", "f16", "f64", "bf16"])
    nx, ny = _log_int(rng, 24, 2048), _log_int(rng, 24, 2048)
    steps = 1
    if kind == "solve":
        # no more work than the largest listed solves: bytes moved, and node updates for FP64
        per_step = 2 * lattice * DTYPE[storage].itemsize * nx * ny
        most = 7e10 / per_step if storage != "f64" else min(7e10 / per_step, 3e7 / (nx * ny))
        steps = 2 * max(4, min(_log_int(rng, 32, 256), int(most / 2)))
    return _one(kind, lattice, nx, ny, geometry, storage, steps, lx=rng.randint(4, max(4, min(64, nx // 3))),
                ly=rng.randint(4, max(4, min(128, ny // 3))), drive="wall" if geometry == "plate" else rng.choice(["body", "wall"]),
                collision=rng.choice(["reg", "reg", "reg", "bgk"]), walls=walls, layout=layout, tau_omega=tau_omega)


def _parameters(lattice, tau_omega):
    """(tau, omega): the period resolves the Stokes layer with four nodes and has 128 steps or more."""
    theta = _table(lattice)[2]
    omega = 2 * math.pi / max(128, math.ceil(8 * math.pi / math.sqrt(2 * theta * tau_omega)))
    return 0.5 + tau_omega / omega, omega


def _instance(case, seed):
    """What one solve of the case is given: tau, omega, u0 and, for ``blocks``, the labels."""
    rng = np.random.default_rng([seed, 9])
    tau, omega = _parameters(case["lattice"], case["tau_omega"] * math.exp(rng.uniform(-0.05, 0.05)))
    u0 = float(rng.uniform(5e-4, 2e-3))
    return dict(case, tau=tau, omega=omega, u0=u0, labels=_labels(case, rng))


def _instances(case, seed):
    """The instances of a batch or a burst: uneven sides, beams and (in a burst) plates."""
    rng = np.random.default_rng(case["mix"])
    out = []
    for k in range(case["count"]):
        serve = case["kind"] == "serve"
        lattice = int(rng.choice([9, 37])) if serve else case["lattice"]
        side = int(round(math.exp(rng.uniform(math.log(case["low"]), math.log(case["high"]))) / 32)) * 32
        side = max(96, side)
        plate = serve and rng.random() < 0.5
        one = _one("solve", lattice, side, side, "plate" if plate else "beam", case["storage"], case["steps"], lx=32,
                   ly=int(rng.choice([8, 16, 32, 64])), drive="wall" if plate else "body",
                   tau_omega=case["tau_omega"] * math.exp(rng.uniform(-1, 1)))
        if serve:  # a request is fitted over a period: it runs for one and a quarter or more
            one["steps"] = max(case["steps"], math.ceil(1.25 * 2 * math.pi / _parameters(lattice, 0.9 * one["tau_omega"])[1]))
        out.append(_instance(one, 1000 * seed + k))
    return out


def _labels(case, rng):
    """Node labels (ny, nx): 0 fluid, 1 body, 2 static wall."""
    nx, ny, reach = case["nx"], case["ny"], 1 if case["lattice"] == 9 else 3
    lab = np.zeros((ny, nx), np.uint8)
    if case["geometry"] == "plate":
        lab[:reach], lab[ny - reach:] = 1, 2
    elif case["geometry"] == "beam":
        x0, y0 = (nx - case["lx"]) // 2, (ny - case["ly"]) // 2
        lab[y0:y0 + case["ly"], x0:x0 + case["lx"]] = 1
    else:  # a body in the left half and an obstacle in the right half, anywhere in it
        for label, left in ((1, 0), (2, nx // 2)):
            w, h = (max(reach, min(case["lx"], nx // 2 - 2 * reach)), max(reach, min(case["ly"], ny - 2 * reach)))
            x0 = left + int(rng.integers(reach, max(reach + 1, nx // 2 - w - reach + 1)))
            y0 = int(rng.integers(0, ny - h + 1))
            lab[y0:y0 + h, x0:x0 + w] = label
    return lab


def work(case):
    """Each population of each fluid node is read once and written once per step; the operations are
    those of the moments, the collision and its source."""
    if case["kind"] in ("batch", "serve"):
        each = [work(i) for i in _instances(case, 0)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    fluid = int((_labels(case, np.random.default_rng(0)) == 0).sum()) * case["steps"]
    return {"bytes": 2 * case["lattice"] * DTYPE[case["storage"]].itemsize * fluid,
            "flops": (500 if case["lattice"] == 37 else 150) * fluid}


# ------------------------------------------------------------------------------------------------
# what a program has in hand, and one pass
# ------------------------------------------------------------------------------------------------

def _geometry(one):
    return dict(kind=GEOMETRY[one["geometry"]], lx=one["lx"], ly=one["ly"], drive=DRIVE[one["drive"]], u0=one["u0"],
                mask=one["labels"] if one["geometry"] == "blocks" else None, eq_order=4 if one["lattice"] == 37 else 2,
                collision=COLLISION[one["collision"]], storage=STORAGE[one["storage"]],
                wall_scheme=WALLS[one["walls"]], layout=LAYOUT[one["layout"]])


class _Server:
    def __init__(self, mode):
        self.handle = L.lbm_server_create(6 << 30, 64)
        L.lbm_server_set_batch_mode(self.handle, mode)

    def __del__(self):
        if getattr(self, "handle", 0):
            L.lbm_server_destroy(self.handle)
            self.handle = 0


def prepare(case, seed):
    if case["kind"] in ("batch", "serve"):
        each = _instances(case, seed)
        descs = [L.make_instance(i["lattice"], i["nx"], i["ny"], i["tau"], i["omega"], i["steps"], **_geometry(i)) for i in each]
        state = {"kind": case["kind"], "each": each, "descs": descs, "steps": case["steps"],
                 "mode": L.LBM_BATCH_PERSISTENT if case["mode"] == "persistent" else L.LBM_BATCH_STREAMS}
        if case["kind"] == "serve":
            state["server"] = _Server(state["mode"])
            # fitted over what follows the first fifth of a period
            state["requests"] = [L.make_request(d, 0.2) for d in descs]
        return state
    one = _instance(case, seed)
    if case["kind"] == "solve":
        return {"kind": "solve", "one": one, "geometry": _geometry(one)}
    sim = L.Simulation(one["lattice"], one["nx"], one["ny"], one["tau"], one["omega"], **_geometry(one))
    flow = _flow(one, seed, L.lbm_info(sim.handle)["pitch"]).to(DTYPE[one["storage"]])
    return {"kind": "step", "sim": sim, "n": _step_index(seed), "in": flow, "out": torch.zeros_like(flow),
            "force": torch.zeros(2, dtype=torch.float64, device=DEVICE)}


def _step_index(seed):
    return 17 + seed % 1000


def _flow(one, seed, pitch):
    """A flow as the library's buffers hold it ([Q][ny][pitch], deviations over w_i s): smooth density
    and velocity waves of the drive's amplitude with some non-equilibrium on top, zero at solids."""
    c, w, theta = _table(one["lattice"])
    nx, ny = one["nx"], one["ny"]
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    rng = np.random.default_rng([seed, 5])
    y, x = torch.meshgrid(torch.arange(ny, device=DEVICE, dtype=torch.float64) / ny,
                          torch.arange(nx, device=DEVICE, dtype=torch.float64) / nx, indexing="ij")
    fields = []
    for amplitude in (0.3, 1.0, 0.5):
        f = torch.zeros_like(x)
        for _ in range(3):
            kx, ky, ph = rng.integers(0, 4), rng.integers(0, 4), rng.uniform(0, 2 * math.pi)
            f += amplitude / 2 * torch.sin(2 * math.pi * (float(kx) * x + float(ky) * y) + ph)
        fields.append(f)
    scale = 1.0 if one["storage"] in ("f16", "bf16") else one["u0"]
    fluid = torch.from_numpy(one["labels"] == 0).to(DEVICE)
    h = torch.zeros((one["lattice"], ny, pitch), dtype=torch.float64, device=DEVICE)
    for i in range(one["lattice"]):
        noise = 0.1 * torch.randn((ny, nx), generator=gen, device=DEVICE, dtype=torch.float64)
        value = fields[0] + (c[i, 0] * fields[1] + c[i, 1] * fields[2]) / theta + noise
        h[i, :, :nx] = scale * value * fluid
    return h


def _as_stored(force, one):
    return torch.from_numpy(force / one["u0"]).to(DTYPE[one["storage"]])


def run(state):
    if state["kind"] == "step":
        L.lbm_step_noalloc(state["sim"].handle, state["n"], state["in"].data_ptr(), state["out"].data_ptr(),
                           state["force"].data_ptr(), torch.cuda.current_stream())
        return {"state": state["out"], "force": state["force"]}
    if state["kind"] == "solve":
        one = state["one"]
        sim = L.lbm_create(one["lattice"], one["nx"], one["ny"], one["tau"], one["omega"], L.make_geometry(**state["geometry"]))
        try:
            L.lbm_step(sim, one["steps"])
            out = {"force": _as_stored(L.lbm_force_history(sim), one)}
            if one["state"]:
                out["state"] = torch.from_numpy(L.lbm_get_state(sim) / one["u0"]).to(DTYPE[one["storage"]])
        finally:
            L.lbm_destroy(sim)
        return out
    if state["kind"] == "batch":
        first = state["descs"][0]
        batch = L.lbm_batch_create(first.lattice, first.geom.storage, first.geom.collision)
        try:
            L.lbm_batch_set_mode(batch, state["mode"])
            slots = [L.lbm_batch_add(batch, d) for d in state["descs"]]
            L.lbm_batch_run(batch, state["steps"])
            L.lbm_batch_synchronize(batch)
            return [_as_stored(L.lbm_force_history(L.lbm_batch_instance(batch, s)), i) for s, i in zip(slots, state["each"])]
        finally:
            L.lbm_batch_destroy(batch)
    server = state["server"].handle
    ids = [L.lbm_server_submit(server, r) for r in state["requests"]]
    out = []
    for rid, one in zip(ids, state["each"]):
        done, result = L.lbm_server_wait(server, rid, 60.0)
        if not done or result["status"] != 2:
            raise RuntimeError(f"request {rid} ended with status {result['status']}")
        fit = torch.tensor([result["f_in"] / one["u0"], result["f_q"] / one["u0"]], dtype=torch.float64)
        out.append({"force": _as_stored(L.lbm_server_force_history(server, rid), one), "fit": fit.to(DTYPE[one["storage"]])})
        L.lbm_server_release(server, rid)
    return out


# ------------------------------------------------------------------------------------------------
# the same in 64 bits with plain torch
# ------------------------------------------------------------------------------------------------

def _table(lattice):
    """(c (Q, 2), w (Q,), theta) as numpy: the rest velocity, then +c and -c of each pair."""
    if lattice == 9:
        pairs = [(1, 0, 1 / 9), (0, 1, 1 / 9), (1, 1, 1 / 36), (1, -1, 1 / 36)]
        w0, theta = 4 / 9, 1 / 3
    else:
        w0, theta = 0.233150669132352, 1 / 1.19697977039307 ** 2
        shells = [(1, 0, 0.107306091542219), (1, 1, 0.0576678598887948), (2, 0, 0.0142082161584507),
                  (2, 2, 0.00101193759267357), (3, 0, 0.000245301027757717), (1, 2, 0.00535304900051377),
                  (1, 3, 0.000283414252994198)]
        pairs = []
        for a, b, w in shells:
            if b == 0:
                pairs += [(a, 0, w), (0, a, w)]
            else:
                pairs += [(a, b, w), (a, -b, w)] + ([(b, a, w), (b, -a, w)] if a != b else [])
    c, w = [(0, 0)], [w0]
    for px, py, wp in pairs:
        c += [(px, py), (-px, -py)]
        w += [wp, wp]
    return np.array(c), np.array(w), theta


class _Exact:
    """The lattice Boltzmann step in FP64 on full-size tensors of deviations g = f - w rho0 (rho0 = 1)."""

    def __init__(self, one):
        self.one = one
        c, w, self.theta = _table(one["lattice"])
        self.Q, self.ny, self.nx = len(w), one["ny"], one["nx"]
        self.order = 4 if one["lattice"] == 37 else 2
        t = dict(dtype=torch.float64, device=DEVICE)
        self.c, self.w = torch.tensor(c.tolist(), **t), torch.tensor(w.tolist(), **t)
        self.ci = c.tolist()
        self.opp = torch.tensor([0] + [i + 1 if i % 2 else i - 1 for i in range(1, self.Q)], device=DEVICE)
        cx, cy = self.c[:, 0], self.c[:, 1]
        self.moments = torch.stack([torch.ones_like(cx), cx, cy, cx * cx, cx * cy, cy * cy])
        self.powers = [(p, q) for p in range(self.order + 1) for q in range(self.order + 1 - p)]
        self.monomials = torch.stack([cx ** p * cy ** q for p, q in self.powers], 1) * self.w[:, None]
        lab = torch.from_numpy(one["labels"]).to(DEVICE)
        self.solid = (lab != 0).reshape(-1)
        # the wall behind a link: the first solid node met walking back from the node to the source
        behind = torch.zeros((self.Q, self.ny, self.nx), dtype=torch.uint8, device=DEVICE)
        for i, (x, y) in enumerate(self.ci):
            for k in range(1, math.gcd(x, y) + 1):
                d = math.gcd(x, y)
                met = torch.roll(lab, (k * y // d, k * x // d), (0, 1))
                behind[i] = torch.where(behind[i] == 0, met, behind[i])
        behind = behind.reshape(self.Q, -1)
        behind[:, self.solid] = 0
        self.nodes = torch.nonzero(behind.any(0)).reshape(-1)
        self.behind = behind[:, self.nodes]
        self.force_sites = self.behind == 1

    def drive(self, n):
        t = n + 0.5
        one = self.one
        return one["u0"] * (math.sin(one["omega"] * t) if one["drive"] == "wall" else one["omega"] * math.cos(one["omega"] * t))

    def maxwellian(self, U):
        """f_eq / (w rho) - 1 of the velocity (U, 0), for every direction."""
        a, b = self.c[:, 0] * U / self.theta, U * U / self.theta
        e = a + (a * a - b) / 2
        if self.order == 4:
            e = e + (a ** 3 - 3 * a * b) / 6 + (a ** 4 - 6 * a * a * b + 3 * b * b) / 24
        return e

    def walls(self, g, pulled, U):
        """Populations that come off the walls (in place of those pulled from solids), and the force."""
        w = self.w[:, None]
        own = g[self.opp][:, self.nodes]
        if self.one["walls"] == "bounce":
            back = own + torch.where(self.force_sites, 2 * w * (self.c[:, :1] * U / self.theta), 0.0)
        else:
            back = torch.zeros_like(own)
            for label, speed in ((1, U), (2, 0.0)):
                at = self.behind == label
                e = self.maxwellian(speed)[:, None]
                share = (w * at).sum(0)
                denominator = (w * (1 + e) * at).sum(0)
                density = torch.where(share > 0, ((own * at).sum(0) - (w * e * at).sum(0)) / torch.where(share > 0, denominator, 1.0), 0.0)
                back = torch.where(at, w * (density + (1 + density) * e), back)
        pulled[:, self.nodes] = torch.where(self.behind > 0, back, pulled[:, self.nodes])
        return -(self.c.T @ ((own + back + 2 * w) * self.force_sites)).sum(1)

    def step(self, g, n):
        one, theta = self.one, self.theta
        tau = one["tau"]
        drive = self.drive(n)
        pulled = torch.stack([torch.roll(g[i].reshape(self.ny, self.nx), (y, x), (0, 1)).reshape(-1) for i, (x, y) in enumerate(self.ci)])
        force = self.walls(g, pulled, drive if one["drive"] == "wall" else 0.0)
        drho, jx, jy, pxx, pxy, pyy = self.moments @ pulled
        rho = 1 + drho
        F = rho * drive if one["drive"] == "body" else torch.zeros_like(rho)
        ux, uy = (jx + F / 2) / rho, jy / rho
        a10, a01 = ux / theta, uy / theta
        b = (ux * ux + uy * uy) / theta
        # coefficients of c_x^p c_y^q: the equilibrium, the even part of the source, the collision
        C = {pq: torch.zeros_like(rho) for pq in self.powers}
        C[0, 0] += drho - rho * b / 2
        linear, square = rho, rho / 2
        if self.order == 4:
            C[0, 0] += rho * b * b / 8
            linear, square = rho - rho * b / 2, rho / 2 - rho * b / 4
            for p in range(4):
                C[p, 3 - p] += rho * (math.comb(3, p) / 6) * a10 ** p * a01 ** (3 - p)
            for p in range(5):
                C[p, 4 - p] += rho * (math.comb(4, p) / 24) * a10 ** p * a01 ** (4 - p)
        C[1, 0] += linear * a10
        C[0, 1] += linear * a01
        C[2, 0] += square * a10 * a10
        C[1, 1] += square * 2 * a10 * a01
        C[0, 2] += square * a01 * a01
        kf = (1 - 0.5 / tau) / theta * F
        S = {(0, 0): -kf * ux, (2, 0): kf * a10, (1, 1): kf * a01}
        if one["collision"] == "reg":
            A = (1 - 1 / tau) / (2 * theta * theta)
            qxx, qxy, qyy = pxx - drho * theta - rho * ux * ux, pxy - rho * ux * uy, pyy - drho * theta - rho * uy * uy
            S[1, 0] = F / (2 * theta)
            S[0, 0] = S[0, 0] - A * theta * (qxx + qyy)
            S[2, 0], S[1, 1], S[0, 2] = S[2, 0] + A * qxx, S[1, 1] + 2 * A * qxy, A * qyy
            for pq, s in S.items():
                C[pq] = C[pq] + s
            out = self.monomials @ torch.stack([C[pq] for pq in self.powers])
        else:
            S[1, 0] = kf
            mix = torch.stack([C[pq] / tau + S.get(pq, 0.0) for pq in self.powers])
            out = (1 - 1 / tau) * pulled + self.monomials @ mix
        out[:, self.solid] = 0.0
        return out, force


def _exact_solve(one):
    ex = _Exact(one)
    g = torch.zeros((ex.Q, ex.ny * ex.nx), dtype=torch.float64, device=DEVICE)
    history = []
    for n in range(one["steps"]):
        g, F = ex.step(g, n)
        history.append(F)
    out = {"force": torch.stack(history) / one["u0"]}
    if one["state"]:
        out["state"] = g.reshape(ex.Q, ex.ny, ex.nx) / one["u0"]
    return out


def _exact_fit(force, one):
    """In-phase and quadrature parts of the force over the steps after a fifth of a period."""
    first = math.ceil(0.2 * 2 * math.pi / one["omega"])
    t = one["omega"] * (np.arange(first, len(force)) + 0.5)
    coef = np.linalg.lstsq(np.stack([np.sin(t), np.cos(t), np.ones_like(t)], 1), force[first:, 0].cpu().numpy(), rcond=None)[0]
    return torch.from_numpy(coef[:2] * (1.0 if one["drive"] == "wall" else -1.0))


def exact(case, seed):
    if case["kind"] == "step":
        one = _instance(case, seed)
        ex = _Exact(one)
        align = 128 // DTYPE[one["storage"]].itemsize
        pitch = -(-one["nx"] // align) * align
        h = _flow(one, seed, pitch).to(DTYPE[one["storage"]]).double()
        unit = (ex.w * (one["u0"] if one["storage"] in ("f16", "bf16") else 1.0))[:, None, None]
        g, F = ex.step((h[:, :, :one["nx"]] * unit).reshape(ex.Q, -1), _step_index(seed))
        h = torch.zeros_like(h)
        h[:, :, :one["nx"]] = g.reshape(ex.Q, one["ny"], one["nx"]) / unit
        return {"state": h, "force": F}
    if case["kind"] == "solve":
        return _exact_solve(_instance(case, seed))
    each = _instances(case, seed)
    solved = [_exact_solve(one)["force"] for one in each]
    if case["kind"] == "batch":
        return solved
    return [{"force": f, "fit": _exact_fit(f, one)} for f, one in zip(solved, each)]
