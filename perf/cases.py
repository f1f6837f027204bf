"""Cases that say how fast the library is in use, each through the calls of a user's program.

Families (a case names its own by "family"):

- ``step``: fixed time steps from a given state, k-space in and out (a program that restores a checkpoint, steps and
  checkpoints again) or real space in and out (a program that draws an initial condition and reads the fields back);
- ``adaptive``: controller-driven step attempts, the way a simulation runs;
- ``ensemble``: several independent simulations advanced by one call;
- ``huchen``: steps with the phase-dependent stiffness (iterated elasticity);
- ``train``: surrogate training steps on consecutive snapshots, the updated weights read back at the end;
- ``infer``: one forward pass of the surrogate.

``exact`` restates the model in 64 bits with plain torch operations.
"""
import math
import random

import numpy as np
import torch

import paper_2609_36100_gb300 as pf
from paper_2609_36100_gb300 import surrogate

# Model constants of the repository's default parameter file (nm, s, GPa, K).
PARAMS = {
    "dx": 0.5, "A_m": 20.0, "A_v": 20.0, "A0_m": 0.0, "A0_v": 0.0, "B_m0": 0.03, "B_v": 0.25, "dBm_dT": 1.0e-4,
    "X_matrix": 0.05, "M0": 0.0025, "Q_act": 250000.0, "T": 973.15, "T0": 973.15, "L": 0.05,
    "kappa": [[0.15, 0.15, 0.15, 0.0, 0.0, 0.0]] * 3, "omega_bar": 0.3, "omega_pair": [0.3] * 3, "pair_eps": 0.01,
    "C11": 250.0, "C12": 160.0, "C44": 120.0,
    "eps_star": [[0.02, 0.004, 0.004, 0.0, 0.0, 0.0], [0.004, 0.02, 0.004, 0.0, 0.0, 0.0],
                 [0.004, 0.004, 0.02, 0.0, 0.0, 0.0]],
    "rtol": 1.0e-4, "atol": 1.0e-8, "h0": 0.5, "h_min": 1.0e-6, "h_max": 100.0, "max_rejects": 10, "safety": 0.9,
    "k1": 0.7, "k2": 0.4, "eta_max": 5.0, "eta_min": 0.2, "eta_reject_min": 0.2,
}
# precipitate stiffness of the phase-contrast cases: C11, C12, C44 raised by 30, 10 and 20 %
CONTRAST = {"el_inhom": 1, "C11_v": 325.0, "C12_v": 176.0, "C44_v": 144.0, "el_max_iter": 20, "el_warm": 1}
RTOL, ATOL = 1.0e-4, 1.0e-8
RHS_PER_STEP = {"euler": 1, "ark2": 3, "ark3": 4, "ark4": 6}


def listed():
    return [
        # the smallest call: one small ensemble-sized grid stepped alone, latency and launches only
        {"name": "ark4-32", "family": "step", "nz": 32, "ny": 32, "nx": 32, "method": "ark4", "precision": "fp32bulk",
         "steps": 4, "dt": 1.0, "nuclei": 4, "elastic": True, "barrier": 0, "space": "hat"},
        # the plain method: 64^3, FP64, first-order semi-implicit fixed steps, real fields in and out
        {"name": "euler-64-fp64", "family": "step", "nz": 64, "ny": 64, "nx": 64, "method": "euler",
         "precision": "fp64", "steps": 10, "dt": 0.5, "nuclei": 8, "elastic": True, "barrier": 0, "space": "real"},
        # a box that is no cube and whose sides are no powers of two, third-order method
        {"name": "ark3-150x108x180", "family": "step", "nz": 150, "ny": 108, "nx": 180, "method": "ark3",
         "precision": "fp32bulk", "steps": 2, "dt": 1.0, "nuclei": 12, "elastic": True, "barrier": 0, "space": "hat"},
        # one snapshot interval of the surrogate's training data: eight fixed steps, the real fields read back
        {"name": "trajectory-128", "family": "step", "nz": 128, "ny": 128, "nx": 128, "method": "ark4",
         "precision": "fp32bulk", "steps": 8, "dt": 1.0, "nuclei": 8, "elastic": True, "barrier": 0, "space": "real"},
        # the FP64 form at the size of the headline workload
        {"name": "ark4-256-fp64", "family": "step", "nz": 256, "ny": 256, "nx": 256, "method": "ark4",
         "precision": "fp64", "steps": 1, "dt": 1.0, "nuclei": 32, "elastic": True, "barrier": 0, "space": "hat"},
        # a large simulation (44 GB of buffers)
        {"name": "ark4-480", "family": "step", "nz": 480, "ny": 480, "nx": 480, "method": "ark4",
         "precision": "fp32bulk", "steps": 1, "dt": 1.0, "nuclei": 126, "elastic": True, "barrier": 0, "space": "hat"},
        # the headline workload: 256^3, adaptive fourth order at rtol 1e-4
        {"name": "adaptive-256", "family": "adaptive", "nz": 256, "ny": 256, "nx": 256, "method": "ark4",
         "precision": "fp32bulk", "attempts": 3, "h0": 1.0, "nuclei": 32, "elastic": True},
        # ensembles over temperature and size: uneven grids, and many small ones
        {"name": "ensemble-uneven", "family": "ensemble", "sides": "64,96,120,128,160,96,64,120", "method": "ark4",
         "precision": "fp32bulk", "t_final": 6.0, "h0": 1.0},
        {"name": "ensemble-small", "family": "ensemble", "sides": "32,48,32,48,32,48,32,48,32,48,32,48,32,48,32,48",
         "method": "ark4", "precision": "fp32bulk", "t_final": 8.0, "h0": 1.0},
        # phase-dependent stiffness at the loose tolerance
        {"name": "huchen-96", "family": "huchen", "nz": 96, "ny": 96, "nx": 96, "method": "ark4",
         "precision": "fp32bulk", "steps": 1, "dt": 1.0, "nuclei": 4, "el_tol": 1e-6},
        # the surrogate at its full size: eight training pairs, and one proposal on a box of other sides
        {"name": "train-128", "family": "train", "nz": 128, "ny": 128, "nx": 128, "C": 32, "modes": 12, "H": 128,
         "L": 4, "bf16": True, "pairs": 8, "lr": 1.0e-3},
        {"name": "infer-160x96x120", "family": "infer", "nz": 160, "ny": 96, "nx": 120, "C": 32, "modes": 12,
         "H": 128, "L": 4, "bf16": True},
    ]


def _smooth(lo, hi):
    out = []
    for n in range(lo, hi + 1, 2):
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            out.append(n)
    return out


def _log_pick(rng, values):
    """One of the sorted values, even over their logarithm."""
    x = math.exp(rng.uniform(math.log(values[0]), math.log(values[-1])))
    return min(values, key=lambda v: abs(math.log(v / x)))


def _box(rng, lo, hi, most):
    values = _smooth(lo, hi)
    while True:
        base = _log_pick(rng, values)
        near = [v for v in values if 0.6 * base <= v <= 1.7 * base]
        s = [base] * 3 if rng.random() < 0.4 else [rng.choice(near) for _ in range(3)]
        if s[0] * s[1] * s[2] <= most:
            return s


def draw(rng):
    family = rng.choice(["step", "step", "step", "adaptive", "ensemble", "huchen", "train", "infer"])
    if family in ("step", "adaptive"):
        precision = rng.choice(["fp32bulk", "fp32bulk", "fp64"])
        most = 256 ** 3 if precision == "fp64" else 480 ** 3
        nz, ny, nx = _box(rng, 24, 480, most)
        n = nz * ny * nx
        method = rng.choice(["ark4", "ark4", "ark3", "ark2", "euler"])
        case = {"family": family, "nz": nz, "ny": ny, "nx": nx, "method": method, "precision": precision,
                "nuclei": max(2, min(126, n // 500000)), "elastic": rng.random() < 0.85}
        if family == "step":
            case["steps"] = 1 if n > 200 ** 3 else rng.choice([1, 2, 4])
            case["dt"] = 0.5 if method in ("euler", "ark2") else 1.0
            case["barrier"] = 1 if rng.random() < 0.15 else 0
            case["space"] = "real" if case["barrier"] or rng.random() < 0.4 else "hat"
        else:
            if method == "euler":
                case["method"] = "ark4"
            case["attempts"] = 1 if n > 200 ** 3 else rng.choice([2, 3])
            case["h0"] = 0.25 if method == "ark2" else 1.0
        return case
    if family == "ensemble":
        small = rng.random() < 0.5
        sides = (32, 48, 60, 64) if small else (64, 80, 96, 120, 128, 144, 160)
        count = rng.randint(6, 16) if small else rng.randint(3, 8)
        return {"family": "ensemble", "sides": ",".join(str(rng.choice(sides)) for _ in range(count)),
                "method": rng.choice(["ark4", "ark4", "ark3"]), "precision": "fp32bulk", "t_final": 4.0, "h0": 1.0}
    if family == "huchen":
        nz, ny, nx = _box(rng, 32, 128, 110 ** 3)
        return {"family": "huchen", "nz": nz, "ny": ny, "nx": nx, "method": rng.choice(["ark4", "ark3"]),
                "precision": rng.choice(["fp32bulk", "fp64"]), "steps": 1, "dt": 1.0, "nuclei": 4,
                "el_tol": rng.choice([1e-6, 1e-4])}
    C, modes, H, L = rng.choice([(32, 12, 128, 4), (32, 8, 128, 4), (16, 6, 64, 4), (32, 8, 64, 3)])
    nz, ny, nx = _box(rng, 32, 160, 128 ** 3)
    case = {"family": family, "nz": nz, "ny": ny, "nx": nx, "C": C, "modes": modes, "H": H, "L": L,
            "bf16": rng.random() < 0.8}
    if family == "train":
        case["pairs"] = rng.choice([1, 2, 4])
        case["lr"] = 1.0e-3
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
DEV = "cuda"


def _params(case, index=0):
    p = dict(PARAMS)
    if not case.get("elastic", True):
        p["eps_star"] = [[0.0] * 6] * 3
    p["barrier"] = int(case.get("barrier", 0))
    if "h0" in case:
        p["h0"] = case["h0"]
    if case["family"] == "huchen":
        p.update(CONTRAST)
        p["el_tol"] = case["el_tol"]
    if case["family"] == "ensemble":  # aging temperatures within 20 K
        p["T"] = p["T0"] + 40.0 * ((index * 0.618034) % 1.0) - 20.0
    return p


def _nuclei(shape, count, rng, rmin, rmax):
    out, tries = [], 0
    while len(out) < count and tries < 20000:
        tries += 1
        r = rng.uniform(rmin, rmax)
        c = [rng.uniform(0, n) for n in shape]
        if all(math.sqrt(sum(min(abs(a - b) % n, n - abs(a - b) % n) ** 2 for a, b, n in zip(c, c2, shape)))
               >= r + r2 + 2.0 for c2, r2 in out):
            out.append((c, r))
    return out


def _fields(shape, count, seed, rmin=4.0, rmax=10.0, grow=0.0, noise=0.0):
    """Spherical nuclei with tanh edges (equilibrium width) of the three variants in a uniform matrix, the composition at
    the precipitate's value inside: real FP64 [4][nz][ny][nx] on the device."""
    rng = random.Random(int(seed))
    top = max(2.0, min(rmax, min(shape) / 5.0))
    ell = math.sqrt(0.15 / 0.3)
    dx = PARAMS["dx"]
    y = torch.zeros((4,) + tuple(shape), dtype=torch.float64, device=DEV)
    for i, (c, r) in enumerate(_nuclei(shape, count, rng, min(rmin, 0.7 * top), top)):
        v = (i + int(seed)) % 3
        r += grow
        ax = []
        for ci, n in zip(c, shape):
            m = int(r) + 24
            i = torch.arange(n, device=DEV) if 2 * m >= n else (torch.arange(-m, m + 1, device=DEV) + int(ci)) % n
            ax.append((i, ((i - ci + n / 2.0) % n - n / 2.0).double()))
        d2 = ax[0][1][:, None, None] ** 2 + ax[1][1][None, :, None] ** 2 + ax[2][1][None, None, :] ** 2
        val = 0.5 * (1.0 - torch.tanh((torch.sqrt(d2) - r) * dx / (math.sqrt(2.0) * ell)))
        ix = (ax[0][0][:, None, None], ax[1][0][None, :, None], ax[2][0][None, None, :])
        y[1 + v][ix] = torch.maximum(y[1 + v][ix], val)
    y[0] = 0.05 + torch.clamp(y[1] + y[2] + y[3], 0.0, 1.0) * (PARAMS["B_v"] - 0.05)
    if noise:
        g = torch.Generator(device=DEV)
        g.manual_seed(int(seed))
        y[0] += noise * torch.randn(y[0].shape, generator=g, dtype=torch.float64, device=DEV)
    return y


def _to_hat(y):
    n = y.shape[-1] * y.shape[-2] * y.shape[-3]
    return torch.stack([torch.fft.rfftn(f) / n for f in y])


def _shape(case):
    return (case["nz"], case["ny"], case["nx"])


def _initial(case, seed):
    noise = 1e-3 if case.get("method") == "euler" else 0.0  # composition noise, as the plain method's start has
    return _fields(_shape(case), case["nuclei"], seed, noise=noise)


def _members(case, seed):
    for i, side in enumerate(int(s) for s in case["sides"].split(",")):
        yield i, _fields((side,) * 3, max(2, side // 8), seed * 1000 + i, 3.0, 6.0)


def _snapshots(case, seed, count):
    """Snapshots [1][count][4][nz][ny][nx] (FP32) of growing nuclei."""
    shape = _shape(case)
    n = max(3, min(8, shape[0] * shape[1] * shape[2] // 100000))
    return torch.stack([_fields(shape, n, seed, 3.0, 6.0, grow=0.25 * t).float() for t in range(count)])[None]


def prepare(case, seed):
    family = case["family"]
    if family in ("train", "infer"):
        shape = _shape(case)
        net = surrogate.new_network(shape, C=case["C"], modes=case["modes"], H=case["H"], L=case["L"],
                                    bf16=case["bf16"], seed=seed)
        if family == "train":
            snaps = _snapshots(case, seed, case["pairs"] + 1)
            net.fit_norm(snaps)
            return {"case": case, "net": net, "snaps": snaps}
        return {"case": case, "net": net, "x": _normalised(_snapshots(case, seed, 1)[0, 0])}
    if family == "ensemble":
        sims, hats = [], []
        for i, y in _members(case, seed):
            sims.append(pf.Simulation(y.shape[1:], _params(case, i), case["method"], case["precision"]))
            hats.append(_to_hat(y))
        return {"case": case, "sims": sims, "hats": hats}
    y = _initial(case, seed)
    sim = pf.Simulation(_shape(case), _params(case), case["method"], case["precision"])
    if case.get("space") == "real":
        return {"case": case, "sim": sim, "y": y, "out": torch.empty_like(y)}
    return {"case": case, "sim": sim, "y": _to_hat(y)}


def _normalised(s):
    mean = s.mean(dim=(1, 2, 3), keepdim=True)
    return ((s - mean) / s.std(dim=(1, 2, 3), keepdim=True).clamp(min=1e-6)).contiguous()


def run(state):
    case = state["case"]
    family = case["family"]
    if family == "train":
        net, s = state["net"], state["snaps"]
        loss = [net.train_pair(s[0, t], s[0, t + 1], case["lr"]) for t in range(case["pairs"])]
        return {"loss": loss, "params": net.params()}
    if family == "infer":
        return state["net"].forward(state["x"])
    if family == "ensemble":
        for sim, y in zip(state["sims"], state["hats"]):
            sim.set_state_hat(y)
            sim.set_time(0.0, case["h0"])
        pf.batch_advance(state["sims"], case["t_final"], RTOL, ATOL)
        return [sim.state_hat() for sim in state["sims"]]
    sim = state["sim"]
    if case.get("space") == "real":
        sim.set_state(state["y"])
        for _ in range(case["steps"]):
            sim.step(case["dt"], want_lte=False)
        return sim.get_state(state["out"])
    sim.set_state_hat(state["y"])
    if family == "adaptive":
        sim.set_time(0.0, case["h0"])
        sim.advance_attempts(case["attempts"], 1e30, RTOL, ATOL)
    else:
        for _ in range(case["steps"]):
            sim.step(case["dt"], want_lte=False)
    return sim.state_hat()


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _rhs_flops(n, elastic=True):
    """Real 3D transforms at 2.5 N log2 N (four in, four out, and three each way for elasticity) and the pointwise
    model, per right-hand side."""
    return (14 if elastic else 8) * 2.5 * n * math.log2(n) + (250 if elastic else 150) * n


def work(case):
    family = case["family"]
    if family in ("train", "infer"):
        n = case["nz"] * case["ny"] * case["nx"]
        C, m, H, L = case["C"], case["modes"], case["H"], case["L"]
        par = 2 * 4 * m ** 3 * C * C * L
        dense = 2 * n * (4 * C + L * C * C + C * H + 4 * H)
        # truncated transforms along x, y, z each way, and the mix
        spectral = L * C * (2 * (4 * n * m + 16 * m * m * n / case["nx"] + 32 * m ** 3 * n / (case["nx"] * case["ny"]))
                            + 8 * 4 * m ** 3 * C)
        if family == "infer":
            return {"bytes": 4 * 8 * n + par * (2 if case["bf16"] else 4), "flops": dense + spectral}
        # weights, two moments and gradients in and out once per pair; states in, weights out to the host
        return {"bytes": case["pairs"] * (4 * 8 * n + 4 * 6 * par) + 4 * par, "flops": case["pairs"] * 3 * (dense + spectral)}
    if family == "ensemble":
        b = f = 0.0
        for side in (int(s) for s in case["sides"].split(",")):
            b += 2 * 4 * 16 * side * side * (side // 2 + 1)
            f += 6 * RHS_PER_STEP[case["method"]] * _rhs_flops(side ** 3)
        return {"bytes": b, "flops": f}
    n = case["nz"] * case["ny"] * case["nx"]
    steps = case.get("steps") or case["attempts"]
    real = case.get("space") == "real"
    flops = steps * RHS_PER_STEP[case["method"]] * _rhs_flops(n, case.get("elastic", True))
    if real:
        flops += 8 * 2.5 * n * math.log2(n)
    if family == "huchen":  # five solves of twelve real transforms for each right-hand side
        flops += steps * RHS_PER_STEP[case["method"]] * 5 * (12 * 2.5 * n * math.log2(n) + 400 * n)
    return {"bytes": 2 * (4 * 8 * n if real else 4 * 16 * n * (case["nx"] // 2 + 1) / case["nx"]), "flops": flops}


def tolerance(case):
    """About four times the distance to exact() that was measured over the listed and some drawn cases."""
    family = case["family"]
    if family == "train":  # Adam's first steps move every weight by about lr, whatever the size of its gradient
        return {"rel": 2e-4, "max": 0.2}
    if family == "infer":
        return {"rel": 1e-4, "max": 8e-3} if case["bf16"] else {"rel": 2e-6, "max": 1e-4}
    if case["precision"] == "fp64":
        return {"rel": 1e-12 if family == "adaptive" else 1e-14, "max": 1e-11}
    return {"rel": 1e-6, "max": 1e-3}


# ---------------------------------------------------------------------------
# the model in 64 bits
# ---------------------------------------------------------------------------
def _tableau(method):
    """(A^E, A^I, b^E, b^I, bt^E, bt^I, embedded order): ImEx Euler, Giraldo, Kelly & Constantinescu (2013), Kennedy &
    Carpenter (2003)."""
    if method == "euler":
        return [[0, 0], [1.0, 0]], [[0, 0], [0, 1.0]], [1.0, 0], [0, 1.0], None, None, 0
    if method == "ark2":
        r2 = math.sqrt(2.0)
        g, a = 1 - 1 / r2, (3 + 2 * r2) / 6
        E = [[0] * 3, [2 - r2, 0, 0], [1 - a, a, 0]]
        b = [1 / (2 * r2), 1 / (2 * r2), g]
        bt = [(4 - r2) / 8, (4 - r2) / 8, 1 / (2 * r2)]
        return E, [[0] * 3, [g, g, 0], b], b, b, bt, bt, 1
    if method == "ark3":
        g = 1767732205903 / 4055673282236
        E = [[0] * 4, [1767732205903 / 2027836641118, 0, 0, 0], [5535828885825 / 10492691773637, 788022342437 / 10882634858940, 0, 0],
             [6485989280629 / 16251701735622, -4246266847089 / 9704473918619, 10755448449292 / 10357097424841, 0]]
        b = [1471266399579 / 7840856788654, -4482444167858 / 7529755066697, 11266239266428 / 11593286722821, g]
        I = [[0] * 4, [g, g, 0, 0], [2746238789719 / 10658868560708, -640167445237 / 6845629431997, g, 0], b]
        bt = [2756255671327 / 12835298489170, -10771552573575 / 22201958757719, 9247589265047 / 10645013368117, 2193209047091 / 5459859503100]
        return E, I, b, b, bt, bt, 2
    E = [[0] * 6, [1 / 2] + [0] * 5, [13861 / 62500, 6889 / 62500] + [0] * 4,
         [-116923316275 / 2393684061468, -2731218467317 / 15368042101831, 9408046702089 / 11113171139209, 0, 0, 0],
         [-451086348788 / 2902428689909, -2682348792572 / 7519795681897, 12662868775082 / 11960479115383, 3355817975965 / 11060851509271, 0, 0],
         [647845179188 / 3216320057751, 73281519250 / 8382639484533, 552539513391 / 3454668386233, 3354512671639 / 8306763924573, 4040 / 17871, 0]]
    b = [82889 / 524892, 0, 15625 / 83664, 69875 / 102672, -2260 / 8211, 1 / 4]
    I = [[0] * 6, [1 / 4, 1 / 4] + [0] * 4, [8611 / 62500, -1743 / 31250, 1 / 4, 0, 0, 0],
         [5012029 / 34652500, -654441 / 2922500, 174375 / 388108, 1 / 4, 0, 0],
         [15267082809 / 155376265600, -71443401 / 120774400, 730878875 / 902184768, 2285395 / 8070912, 1 / 4, 0], b]
    bt = [4586570599 / 29645900160, 0, 178811875 / 945068544, 814220225 / 1159782912, -3700637 / 11593932, 61727 / 225920]
    return E, I, b, b, bt, bt, 3


def _cubic(c, e):
    """Cubic Hooke's law on (xx, yy, zz, yz, xz, xy) tensor components."""
    tr = e[0] + e[1] + e[2]
    return [(c[0] - c[1]) * e[i] + c[1] * tr for i in range(3)] + [2 * c[2] * e[i] for i in range(3, 6)]


def _cubic_inv(c):
    d = (c[0] - c[1]) * (c[0] + 2 * c[1])
    return (c[0] + c[1]) / d, -c[1] / d, 1 / (2 * c[2])


class _Model:
    def __init__(self, shape, p):
        self.shape, self.p = shape, p
        self.n = shape[0] * shape[1] * shape[2]
        m = [torch.fft.fftfreq(s, dtype=torch.float64, device=DEV) for s in shape[:2]]
        m.append(torch.fft.rfftfreq(shape[2], dtype=torch.float64, device=DEV))
        kz, ky, kx = (2 * math.pi / p["dx"] * t for t in m)
        # the Nyquist wave number is +pi/dx
        self.k = [kx[None, None, :], torch.where(ky == ky.min(), -ky, ky)[None, :, None],
                  torch.where(kz == kz.min(), -kz, kz)[:, None, None]]
        self.k2 = self.k[0] ** 2 + self.k[1] ** 2 + self.k[2] ** 2
        self.M = p["M0"] * math.exp(-p["Q_act"] / 8.314462618 * (1 / p["T"] - 1 / p["T0"]))
        self.Bm = p["B_m0"] + p["dBm_dT"] * (p["T"] - p["T0"])
        self.lam = [-2 * p["A_m"] * self.M * self.k2] + [-p["L"] * p["kappa"][v][0] * self.k2 for v in range(3)]
        self.elastic = any(any(e) for e in p["eps_star"])
        self.prev = None

    def to_r(self, y):
        return [torch.fft.irfftn(f * self.n, s=self.shape) for f in y]

    def to_k(self, f):
        return torch.fft.rfftn(f) / self.n

    def normal(self):
        k = torch.sqrt(self.k2)
        k[0, 0, 0] = 1.0
        n = [q / k for q in self.k]
        return n

    def acoustic_solve(self, c, n, b):
        """(n.C.n)^-1 b by cofactors, C cubic."""
        c11, c12, c44 = c
        a = [c44 + (c11 - c44) * q * q for q in n]
        d, e, f = (c12 + c44) * n[0] * n[1], (c12 + c44) * n[0] * n[2], (c12 + c44) * n[1] * n[2]
        A = [[a[1] * a[2] - f * f, e * f - d * a[2], d * f - a[1] * e], [None, a[0] * a[2] - e * e, d * e - a[0] * f],
             [None, None, a[0] * a[1] - d * d]]
        det = a[0] * A[0][0] + d * A[0][1] + e * A[0][2]
        return [sum(A[min(i, j)][max(i, j)] * b[j] for j in range(3)) / det for i in range(3)]

    def potential(self, h):
        p = self.p
        n = self.normal()
        c = (p["C11"], p["C12"], p["C44"])
        hk = [self.to_k(f) for f in h]
        for f in hk:
            f[0, 0, 0] = 0
        sig = [_cubic(c, e) for e in p["eps_star"]]

        def dot(s, n):
            return [s[0] * n[0] + s[5] * n[1] + s[4] * n[2], s[5] * n[0] + s[1] * n[1] + s[3] * n[2], s[4] * n[0] + s[3] * n[1] + s[2] * n[2]]

        t = [sum(sig[q][i] * hk[q] for q in range(3)) for i in range(6)]  # sum of sigma*_q h_q
        u = self.acoustic_solve(c, n, dot(t, n))
        out = []
        for v in range(3):
            e = p["eps_star"][v]
            first = sum(e[i] * t[i] for i in range(3)) + 2 * sum(e[i] * t[i] for i in range(3, 6))
            s = dot(sig[v], n)
            out.append(torch.fft.irfftn((first - sum(s[i] * u[i] for i in range(3))) * self.n, s=self.shape))
        return out

    def iterate(self, h):
        """The iterated elastic solve around the mean of the two stiffnesses, started from the last solve's strain."""
        p = self.p
        cm, cv = (p["C11"], p["C12"], p["C44"]), (p["C11_v"], p["C12_v"], p["C44_v"])
        c0 = tuple(0.5 * (a + b) for a, b in zip(cm, cv))
        sm, sv = _cubic_inv(cm), _cubic_inv(cv)
        H = h[0] + h[1] + h[2]
        c = _cubic_inv([(1 - H) * a + H * b for a, b in zip(sm, sv)])
        e0 = [sum(h[v] * p["eps_star"][v][i] for v in range(3)) for i in range(6)]
        scale = max(float(q.abs().max()) for q in e0)
        n = self.normal()
        keep = torch.ones_like(self.k2)
        keep[0, 0, 0] = 0
        keep[self.shape[0] // 2], keep[:, self.shape[1] // 2], keep[:, :, self.shape[2] // 2] = 0, 0, 0

        def green(tau):
            t = [self.to_k(f) * keep for f in tau]
            w = self.acoustic_solve(c0, n, [t[0] * n[0] + t[5] * n[1] + t[4] * n[2], t[5] * n[0] + t[1] * n[1] + t[3] * n[2], t[4] * n[0] + t[3] * n[1] + t[2] * n[2]])
            return [torch.fft.irfftn(0.5 * (n[i] * w[j] + n[j] * w[i]) * self.n, s=self.shape) for i, j in ((0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1))]

        def mean_strain(eu):
            r = [float(q.mean()) for q in _cubic(c, [a - b for a, b in zip(e0, eu)])]
            s = _cubic_inv([float(q.mean()) for q in c])
            tr = r[0] + r[1] + r[2]
            return [(s[0] - s[1]) * r[i] + s[1] * tr for i in range(3)] + [s[2] * r[i] for i in range(3, 6)]

        t0 = _cubic(c0, e0)
        it = 0
        eu = self.prev
        if eu is None:
            eu, it = green(t0), 1
        eb = mean_strain(eu)
        while it < p["el_max_iter"]:
            s = _cubic([a - b for a, b in zip(c, c0)], [b + u - e for b, u, e in zip(eb, eu, e0)])
            new = green([a - b for a, b in zip(t0, s)])
            change = max(float((a - b).abs().max()) for a, b in zip(new, eu))
            eu, it = new, it + 1
            eb = mean_strain(eu)
            if not change > p["el_tol"] * scale:
                break
        self.prev = eu
        s = _cubic(c, [b + u - e for b, u, e in zip(eb, eu, e0)])
        d = [b - a for a, b in zip(sm, sv)]
        half = 0.5 * (d[0] * (s[0] ** 2 + s[1] ** 2 + s[2] ** 2) + 2 * d[1] * (s[0] * s[1] + s[1] * s[2] + s[0] * s[2]) + 2 * d[2] * (s[3] ** 2 + s[4] ** 2 + s[5] ** 2))
        return [-sum(s[i] * e[i] for i in range(3)) - 2 * sum(s[i] * e[i] for i in range(3, 6)) - half for e in p["eps_star"]]

    def rhs(self, y):
        p = self.p
        X, *f = self.to_r(y)
        h = [q ** 3 * (6 * q * q - 15 * q + 10) for q in f]
        H = h[0] + h[1] + h[2]
        iv, im = 1 / (2 * p["A_v"]), 1 / (2 * p["A_m"])
        mu = (X - H * p["B_v"] - (1 - H) * self.Bm) / (H * iv + (1 - H) * im)
        drive = p["A0_v"] + p["A_v"] * (mu * iv) ** 2 - p["A0_m"] - p["A_m"] * (mu * im) ** 2 - mu * (mu * iv + p["B_v"] - mu * im - self.Bm)
        if self.elastic:
            e = self.iterate(h) if p.get("el_inhom") else self.potential(h)
        w12, w13, w23 = p["omega_pair"]
        w = [[0, w12, w13], [w12, 0, w23], [w13, w23, 0]]
        out = [-self.M * self.k2 * self.to_k(mu - 2 * p["A_m"] * X)]
        for v in range(3):
            if p["barrier"]:
                g = p["omega_bar"] * (1 - 2 * (f[0] + f[1] + f[2]))
            else:
                g = 2 * p["omega_bar"] * f[v] * (1 - f[v]) * (1 - 2 * f[v])
            for q in range(3):
                if q != v:
                    g = g + w[v][q] * torch.clamp(f[v] * f[q] / p["pair_eps"], -1, 1) * f[q]
            hp = 30 * f[v] ** 2 * (1 - f[v]) ** 2
            g = g + hp * (drive + e[v]) if self.elastic else g + hp * drive
            out.append(-p["L"] * self.to_k(g))
        return out

    def step(self, y, dt, method, want_lte=False):
        E, I, bE, bI, tE, tI, _ = _tableau(method)
        Z, F = [], []
        s = len(bE)
        for i in range(s):
            gamma = dt * I[i][i]
            z = []
            for f in range(4):
                r = y[f].clone()
                for j in range(i):
                    if I[i][j]:
                        r += dt * I[i][j] * self.lam[f] * Z[j][f]
                    if E[i][j]:
                        r += dt * E[i][j] * F[j][f]
                z.append(r / (1 - gamma * self.lam[f]) if gamma else r)
            Z.append(z)
            used = bE[i] or any(E[k][i] for k in range(i + 1, s)) or (tE and tE[i])
            F.append(self.rhs(z) if used else None)
        new, lte = [], []
        for f in range(4):
            r, e = y[f].clone(), torch.zeros_like(y[f])
            for i in range(s):
                if bI[i]:
                    r += dt * bI[i] * self.lam[f] * Z[i][f]
                if bE[i]:
                    r += dt * bE[i] * F[i][f]
                if want_lte and bI[i] != tI[i]:
                    e += dt * (bI[i] - tI[i]) * self.lam[f] * Z[i][f]
                if want_lte and bE[i] != tE[i]:
                    e += dt * (bE[i] - tE[i]) * F[i][f]
            new.append(r)
            lte.append(e)
        if self.p["barrier"]:
            new = new[:1] + [self.to_k(torch.clamp(q, 0, 1)) for q in self.to_r(new)[1:]]
        if not want_lte:
            return new
        sq = sum(float(((a / (RTOL * b.abs() + ATOL)) ** 2).sum()) for a, b in zip(self.to_r(lte), self.to_r(y)))
        return new, math.sqrt(sq / (4 * self.n))

    def advance(self, y, h, method, t_final, attempts):
        p = self.p
        q = _tableau(method)[6] + 1
        t, last, rejected = 0.0, 1.0, False
        for _ in range(attempts):
            if not t < t_final * (1 - 1e-14):
                break
            h = min(h, t_final - t)
            new, e = self.step(y, h, method, True)
            if e <= 1.0:
                y, t = new, t + h
                e = max(e, 1e-10)
                h *= min(1.0 if rejected else p["eta_max"], max(p["eta_min"], p["safety"] * e ** (-p["k1"] / q) * last ** (p["k2"] / q)))
                last, rejected = e, False
            else:
                h *= max(p["eta_reject_min"], p["safety"] * e ** (-1 / q))
                rejected = True
            h = min(max(h, p["h_min"]), p["h_max"])
        return y


def _exact_net(case, theta):
    """The network as a function of (theta, x), both FP64; theta a flat leaf tensor in the library's order."""
    nz, ny, nx = _shape(case)
    C, m, H, L = case["C"], case["modes"], case["H"], case["L"]
    K = 4 * m ** 3
    sizes = [("P", (C, 4)), ("p", (C,))]
    for l in range(L):
        sizes += [("W%d" % l, (K, C, C, 2)), ("V%d" % l, (C, C)), ("v%d" % l, (C,))]
    sizes += [("Q1", (H, C)), ("q1", (H,)), ("Q2", (4, H)), ("q2", (4,))]
    iy = torch.tensor(list(range(m)) + list(range(ny - m, ny)), device=DEV)
    iz = torch.tensor(list(range(m)) + list(range(nz - m, nz)), device=DEV)

    def part(t):
        out, o = {}, 0
        for name, s in sizes:
            out[name] = t[o:o + math.prod(s)].reshape(s)
            o += math.prod(s)
        return out

    def forward(t, x):
        w = part(t)
        col = lambda b: b[:, None, None, None]  # noqa: E731
        a = torch.einsum("cf,fzyx->czyx", w["P"], x) + col(w["p"])
        for l in range(L):
            W = w["W%d" % l]
            if case["bf16"]:  # spectral weights are used in bf16, gradients pass to the FP32 copy
                W = W + (W.detach().float().bfloat16().double() - W.detach())
            A = torch.fft.rfftn(a, dim=(1, 2, 3))[:, iz][:, :, iy][..., :m].reshape(C, K)
            O = torch.einsum("kcd,dk->ck", torch.view_as_complex(W.contiguous()), A).reshape(C, 2 * m, 2 * m, m)
            full = torch.zeros((C, nz, ny, m), dtype=torch.complex128, device=DEV)
            full = full.index_put((torch.arange(C, device=DEV)[:, None, None], iz[None, :, None], iy[None, None, :]), O)
            s = torch.fft.ifftn(full, dim=(1, 2), norm="forward")
            # along x: Re sum of w_k s_k e^{2 pi i k x / nx} / N, w = 1 for k = 0 and 2 otherwise
            ph = 2 * math.pi * torch.outer(torch.arange(m, device=DEV), torch.arange(nx, device=DEV)).remainder(nx).double() / nx
            wk = torch.full((m, 1), 2.0, dtype=torch.float64, device=DEV)
            wk[0] = 1.0
            s = (torch.einsum("czyk,kx->czyx", s.real, wk * torch.cos(ph)) - torch.einsum("czyk,kx->czyx", s.imag, wk * torch.sin(ph))) / (nz * ny * nx)
            z = torch.einsum("cd,dzyx->czyx", w["V%d" % l], a) + col(w["v%d" % l]) + s
            a = torch.nn.functional.gelu(z) if l < L - 1 else z
        h = torch.nn.functional.gelu(torch.einsum("hc,czyx->hzyx", w["Q1"], a) + col(w["q1"]))
        return torch.einsum("fh,hzyx->fzyx", w["Q2"], h) + col(w["q2"])

    return forward


def exact(case, seed):
    family = case["family"]
    if family in ("train", "infer"):
        net = surrogate.new_network(_shape(case), C=case["C"], modes=case["modes"], H=case["H"], L=case["L"],
                                    bf16=case["bf16"], seed=seed)
        theta = torch.from_numpy(net.params()).to(DEV).double()  # the same starting weights
        net.close()
        forward = _exact_net(case, theta)
        if family == "infer":
            return forward(theta, _normalised(_snapshots(case, seed, 1)[0, 0]).double())
        s = _snapshots(case, seed, case["pairs"] + 1)[0].double()
        stat = lambda t: (t.mean(dim=(0, 2, 3, 4)), t.std(dim=(0, 2, 3, 4), unbiased=False))  # noqa: E731
        mean, sd = stat(s[:-1])
        dsd = stat(s[1:] - s[:-1])[1]
        mean, sd, dsd = mean[:, None, None, None], torch.clamp(sd, min=1e-6)[:, None, None, None], torch.clamp(dsd, min=1e-9)[:, None, None, None]
        m, v = torch.zeros_like(theta), torch.zeros_like(theta)
        loss = []
        for t in range(case["pairs"]):
            leaf = theta.detach().requires_grad_(True)
            x, tgt = (s[t] - mean) / sd, (s[t + 1] - s[t]) / dsd
            e = ((forward(leaf, x) - tgt) ** 2).mean()
            g, = torch.autograd.grad(e, leaf)
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            theta = theta - case["lr"] * (m / (1 - 0.9 ** (t + 1))) / (torch.sqrt(v / (1 - 0.999 ** (t + 1))) + 1e-8)
            loss.append(float(e.detach()))
        return {"loss": loss, "params": theta}
    if family == "ensemble":
        out = []
        for i, y in _members(case, seed):
            mod = _Model(tuple(y.shape[1:]), _params(case, i))
            out.append(torch.stack(mod.advance(list(_to_hat(y)), case["h0"], case["method"], case["t_final"], 100)))
        return out
    if case["nz"] * case["ny"] * case["nx"] > 300 ** 3:
        return None  # over 20 s
    y = list(_to_hat(_initial(case, seed)))
    mod = _Model(_shape(case), _params(case))
    if family == "adaptive":
        return torch.stack(mod.advance(y, case["h0"], case["method"], 1e30, case["attempts"]))
    for _ in range(case["steps"]):
        y = mod.step(y, case["dt"], case["method"])
    return torch.stack(mod.to_r(y) if case.get("space") == "real" else y)
