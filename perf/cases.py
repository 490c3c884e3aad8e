"""The work that is timed: the calls that a program makes on this library, over their range.

A case is one pass of a program's loop through the public binding.  Kinds:

  plain    load the orbitals, apply the exchange to every pair, take W and E_x
           (the untruncated operator: a reference run, or a small molecule)
  step     one outer step of the double SCF loop: orthonormalise, localise,
           screen, exchange, build ACE, apply it to a block of trial functions
  apply    one inner step: the kept projector applied to a block on the device
  serve    resident systems of one request server, each rebuilt once and then
           applied twice, host arrays in and out
  batch    independent systems run together

Orbitals are sums of band-limited Gaussians at the density of liquid water
(as `synth` makes them for the serving stream), mixed by a random orthogonal
matrix so that they start delocalised, made on the device from the seed.

A mixed-precision context computes its grids in 32 bits, and what it returns
in 64-bit arrays carries no more than that: the program that chose it keeps
the results in 32 bits.  FP64 contexts' results are kept as they come.
"""
import math

import numpy as np
import torch

from paper_1801_09263_gb300 import binding as lace

BOHR3_PER_ORBITAL = 30.0 * 1.8897261**3 / 4.0  # water: 30 A^3 a molecule, 4 occupied orbitals
SIZES = [n for n in range(24, 129) if all(p == 1 for p in [n // math.gcd(n, (2**7) * (3**4) * (5**3))])]
S_THR = 1e-3


def _case(name, kind, shape, n_occ, n_extra=0, precision="mixed", block=32, screened=False, shear=0.0):
    return {"name": name, "kind": kind, "n1": shape[0], "n2": shape[1], "n3": shape[2], "n_occ": n_occ,
            "n_extra": n_extra, "precision": precision, "block": block, "screened_kernel": screened, "shear": shear}


def listed():
    return [
        # the smallest: 8 orbitals on 24^3 in FP64 with W read back (a reference evaluation)
        _case("plain_24_fp64", "plain", (24, 24, 24), 8, precision="fp64"),
        # the smallest system of an uneven batch, run by itself
        _case("step_32", "step", (32, 32, 32), 16),
        # a small molecule or a small water cluster, and the same on an odd grid
        _case("step_48", "step", (48, 48, 48), 64),
        _case("step_45_odd", "step", (45, 45, 45), 60),
        # the 64-molecule water box: the ordinary step
        _case("step_72", "step", (72, 72, 72), 256, block=256),
        # an orthorhombic box (a solute in water) with the screened kernel of HSE
        _case("step_hse_slab", "step", (72, 80, 64), 192, block=64, screened=True, shear=0.1),
        # empty states in the projection set: every pair with one is computed
        _case("step_96_extra", "step", (96, 96, 96), 256, n_extra=128, block=8),
        # a dense grid of the serving range
        _case("step_120", "step", (120, 120, 120), 320),
        # the localised step in FP64
        _case("step_48_fp64", "step", (48, 48, 48), 32, precision="fp64"),
        # the inner loop: one block of a Davidson step
        _case("apply_72", "apply", (72, 72, 72), 256, block=64),
        # four resident systems of a request server
        _case("serve_4", "serve", (48, 48, 48), 48, block=32),
        # twelve uneven systems run together
        _case("batch_12", "batch", (32, 64, 0), 12),
    ]


def _cell(case):
    """The box at water density; `shear` makes its edges uneven (1 : 1 + shear : 1 - shear)."""
    edges = np.array([1.0, 1.0 + case["shear"], 1.0 - case["shear"]])
    return edges * (case["n_occ"] * BOHR3_PER_ORBITAL / edges.prod()) ** (1.0 / 3.0)


def _shape(case):
    return (case["n1"], case["n2"], case["n3"])


def _kept(n):
    """Pairs kept at S_THR at this density: about 7.4 an orbital in a large box."""
    return min(n * (n + 1) // 2, round(7.4 * n))


def _sub(case):
    """The systems of a serve or batch case, as step cases."""
    rng = np.random.default_rng(case["n_occ"] * 1000 + case["n1"])
    out = []
    if case["kind"] == "serve":  # one grid, orbital counts around n_occ
        for k in range(4):
            n = max(8, int(case["n_occ"] * (0.7 + 0.2 * k)))
            out.append(_case("", "step", _shape(case), n, block=case["block"]))
    else:  # n_occ systems on cubic grids from n1 to n2
        sizes = [n for n in SIZES if case["n1"] <= n <= case["n2"]]
        for k in range(case["n_occ"]):
            n = sizes[(k * len(sizes)) // case["n_occ"]]
            out.append(_case("", "step", (n, n, n), int(round(16 * 8 ** rng.uniform())), block=0))
    return out


def work(case):
    """Bytes: orbitals and functions in, results out.  Operations: the FFTs of the pairs (two real
    densities a complex transform) and the contractions over the grid."""
    if case["kind"] in ("serve", "batch"):
        total = {"bytes": 0.0, "flops": 0.0}
        for c in _sub(case):
            w = work(c)
            extra = work(dict(c, kind="apply")) if case["kind"] == "serve" else {"bytes": 0.0, "flops": 0.0}
            for k in total:
                total[k] += w[k] + extra[k]
        return total
    n, e, b = case["n_occ"], case["n_extra"], case["block"]
    ng = float(case["n1"] * case["n2"] * case["n3"])
    p = n + e
    apply_flops = 4.0 * p * b * ng
    if case["kind"] == "apply":
        word = 4
        return {"bytes": word * p * ng + 8.0 * b * ng + (8 + word) * b * ng, "flops": apply_flops}
    pairs = (n * (n + 1) // 2 if case["kind"] == "plain" else _kept(n)) + n * e
    flops = pairs * (5.0 * ng * math.log2(ng) + 6.0 * ng) + n * n * ng
    if case["kind"] == "plain":
        return {"bytes": 16.0 * n * ng, "flops": flops + 2.0 * n * n * ng}
    flops += (2.0 * n * n + n * n + 4.0 * p * p + 4.0 * n * e) * ng + apply_flops
    return {"bytes": 8.0 * p * ng + (16.0 + 4.0) * b * ng, "flops": flops}


def draw(rng):
    """The same kinds over their ranges: 8 to 384 orbitals, 24 to 128 points an axis, cubic and not."""
    while True:
        kind = rng.choice(["plain", "step", "step", "step", "step", "apply", "apply"])
        fp64 = kind == "plain" or (kind == "step" and rng.random() < 0.15)
        most = 16 if kind == "plain" else 48 if fp64 else 384
        n = round(math.exp(rng.uniform(math.log(8 if kind == "plain" else 16), math.log(most))))
        shear = 0.0 if rng.random() < 0.5 else round(rng.uniform(0.03, 0.2), 3)
        extra = round(n * rng.uniform(0.1, 0.4)) if kind != "plain" and rng.random() < 0.25 else 0
        block = round(math.exp(rng.uniform(math.log(4), math.log(256))))
        case = _case("", kind, (0, 0, 0), n, extra, "fp64" if fp64 else "mixed", min(block, n + extra),
                     rng.random() < 0.3, shear)
        spacing = rng.uniform(0.24, 0.40)
        for key, edge in zip(("n1", "n2", "n3"), _cell(case)):
            at = min(range(len(SIZES)), key=lambda i: abs(SIZES[i] - edge / spacing))
            case[key] = SIZES[at]
        del case["name"]
        top = 72 if fp64 else 128
        if max(_shape(case)) > top or case["n1"] * case["n2"] * case["n3"] < 24**3:
            continue
        if work(case)["flops"] <= (6e10 if fp64 else 2.5e12):
            return case


# ------------------------------------------------------------------ inputs

def _orbitals(case, n, rng, mix, device="cuda"):
    """n raw orbitals [n, n1, n2, n3] float64: 4 Gaussians each around one of 3n/4 centres."""
    cell, shape = _cell(case), _shape(case)
    ecut = _ecut(case)
    centres = rng.uniform(size=(max(1, 3 * n // 4), 3)) * cell
    pos = centres[np.repeat(np.arange(n), 4) % len(centres)] + rng.normal(0.0, 0.5, size=(4 * n, 3))
    alpha = rng.uniform(0.5, 2.0, size=4 * n)
    coef = rng.uniform(-1.0, 1.0, size=4 * n)
    f = []
    for a in range(3):
        m = np.arange(1, int(math.sqrt(2.0 * ecut) * cell[a] / (2.0 * math.pi)) + 1)
        g = torch.tensor(2.0 * math.pi * m / cell[a], device=device)
        x = torch.arange(shape[a], device=device, dtype=torch.float64) * (cell[a] / shape[a])
        al = torch.tensor(alpha, device=device)
        d = x[None, :] - torch.tensor(pos[:, a], device=device)[:, None]
        w = torch.exp(-g[None, :] ** 2 / (4.0 * al[:, None]))
        s = 1.0 + 2.0 * torch.einsum("tm,tmx->tx", w, torch.cos(g[None, :, None] * d[:, None, :]))
        f.append((s * (torch.sqrt(math.pi / al) / cell[a])[:, None]).view(n, 4, shape[a]))
    f[0] = f[0] * torch.tensor(coef, device=device).view(n, 4, 1)
    xy = torch.einsum("otx,oty->oxyt", f[0], f[1]).reshape(n, shape[0] * shape[1], 4)
    phi = torch.bmm(xy, f[2])
    del xy
    phi = phi.view(n, -1)
    if mix:
        q = torch.tensor(np.linalg.qr(rng.standard_normal((n, n)))[0], device=device)
        phi = q.T @ phi
    return phi.view((n,) + shape)


def _ecut(case):
    return float(min(40.0, 0.45 * min((math.pi * k / a) ** 2 for k, a in zip(_shape(case), _cell(case)))))


def _inputs(case, seed, device="cuda"):
    """The raw orbitals (extras last) and a block of trial functions: orbitals that have moved a little."""
    rng = np.random.default_rng(seed)
    phi = _orbitals(case, case["n_occ"], rng, True, device)
    if case["n_extra"]:
        phi = torch.cat([phi, _orbitals(case, case["n_extra"], rng, False, device)])
    psi = None
    if case["kind"] != "plain" and case["block"]:
        b = case["block"]
        psi = phi[torch.arange(b) % len(phi)]
        norm = torch.sqrt(_dv(case) * (psi * psi).sum(dim=(1, 2, 3), keepdim=True))
        psi = psi / norm
        psi += 0.05 * torch.roll(psi, 1, 1)
    return phi, psi


def _dv(case):
    return float(np.prod(_cell(case))) / (case["n1"] * case["n2"] * case["n3"])


def _kernel_args(case):
    return (lace.KERNEL_ERFC, 0.11, 0.25) if case["screened_kernel"] else (lace.KERNEL_COULOMB, 0.0, 1.0)


# ------------------------------------------------------------------ the calls

def _context(case, stream):
    ctx = lace.Lace(0, lace.LACE_FP64 if case["precision"] == "fp64" else lace.LACE_MIXED)
    ctx.set_stream(stream.cuda_stream)
    ctx.set_cell(_cell(case), _shape(case), _ecut(case))
    ctx.set_kernel(*_kernel_args(case))
    return ctx


def _step(s):
    ctx, case = s["ctx"], s["case"]
    ctx.load_orbitals_dev(s["phi"], case["n_occ"], case["n_extra"], True)
    ctx.localize(2)
    n_pairs = ctx.screen(S_THR)
    _, ex = ctx.apply_exchange(want_W=False)
    ctx.build_ace()
    return n_pairs, ex


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        srv = lace.Server(0, lace.LACE_MIXED, slots=4)
        systems = []
        for k, c in enumerate(_sub(case)):
            phi, psi = _inputs(c, seed * 64 + k)
            sid = srv.add_system(_cell(c), _shape(c), _ecut(c), c["n_occ"], 0, S_THR)
            hold = [t.cpu().pin_memory() for t in (phi, psi)]
            out = torch.empty_like(hold[1]).pin_memory()
            systems.append((sid, hold[0].numpy(), hold[1].numpy(), out.numpy(), (hold, out)))
        return {"case": case, "srv": srv, "systems": systems}
    if kind == "batch":
        subs = _sub(case)
        b = lace.Batch([(_cell(c), _shape(c), _ecut(c), c["n_occ"], S_THR) for c in subs])
        hold = []
        for k, c in enumerate(subs):
            hold.append(_inputs(c, seed * 64 + k)[0].cpu().pin_memory())
            b.set_orbitals(k, hold[-1].numpy())
        b.run()  # the program's first run chooses the launch shape, its second captures the graph
        return {"case": case, "batch": b, "hold": hold}
    phi, psi = _inputs(case, seed)
    stream = torch.cuda.Stream()
    s = {"case": case, "phi": phi, "psi": psi, "stream": stream, "ctx": _context(case, stream)}
    if psi is not None:
        s["out"] = torch.empty_like(psi)
    torch.cuda.synchronize()
    if kind == "apply":  # the projector of the current outer step
        _step(s)
        s["phi"] = None
    return s


def _kept_bits(case, v):
    return v if case["precision"] == "fp64" else v.to(torch.float32) if isinstance(v, torch.Tensor) else np.float32(v)


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "serve":
        srv, out = s["srv"], {}
        built = [srv.submit_rebuild(sid, phi) for sid, phi, _, _, _ in s["systems"]]
        ex = [srv.poll(r) for r in built]
        for _ in range(2):
            sent = [srv.submit_apply(sid, psi, out=to) for sid, _, psi, to, _ in s["systems"]]
            done = [srv.poll(r) for r in sent]
        for k, (r, a) in enumerate(zip(ex, done)):
            if r["status"] or a["status"]:
                raise RuntimeError(r["error"] or a["error"])
            out["ex%d" % k] = np.float32(r["ex"])
            out["kpsi%d" % k] = torch.from_numpy(a["out"]).to(torch.float32)
        return out
    if kind == "batch":
        ex, status = s["batch"].run()
        if status.any():
            raise RuntimeError("an instance failed: %s" % status)
        mats = [s["batch"].context(k).get_matrix(lace.MAT_PAIR_ENERGY) for k in range(len(ex))]
        return {"ex": ex.astype(np.float32), "pair_e": [m.astype(np.float32) for m in mats]}
    ctx = s["ctx"]
    with torch.cuda.stream(s["stream"]):
        if kind == "plain":
            ctx.load_orbitals_dev(s["phi"], case["n_occ"], 0, True)
            W, ex = ctx.apply_exchange()
            return {"W": W, "ex": ex}
        if kind == "apply":
            ctx.apply_ace_dev(s["psi"], s["out"])
            return {"kpsi": _kept_bits(case, s["out"]), "e_block": _kept_bits(case, ctx.ace_energy())}
        n_pairs, ex = _step(s)
        ctx.apply_ace_dev(s["psi"], s["out"])
        return {"n_pairs": n_pairs, "ex": _kept_bits(case, ex), "kpsi": _kept_bits(case, s["out"])}


# ------------------------------------------------------------------ the same in 64 bits

def _inv_sqrt(a):
    w, v = torch.linalg.eigh(a)
    return (v / torch.sqrt(w)) @ v.T


def _lowdin(x, dv):
    return _inv_sqrt(dv * (x @ x.T)) @ x


def _k_table(case, device):
    cell, shape = _cell(case), _shape(case)
    g = [2.0 * math.pi * torch.fft.fftfreq(k, 1.0 / k, device=device, dtype=torch.float64) / a for k, a in zip(shape, cell)]
    gz = g[2][: shape[2] // 2 + 1].abs()
    g2 = g[0][:, None, None] ** 2 + g[1][None, :, None] ** 2 + gz[None, None, :] ** 2
    safe = torch.where(g2 > 0, g2, torch.ones_like(g2))
    if case["screened_kernel"]:
        _, omega, fraction = _kernel_args(case)
        k = 4.0 * math.pi / safe * (1.0 - torch.exp(-safe / (4.0 * omega * omega)))
        return fraction * torch.where(g2 > 0, k, torch.full_like(k, math.pi / omega**2))
    return torch.where(g2 > 0, 4.0 * math.pi / safe, torch.zeros_like(g2))


def _exchange(case, psi, n, pairs):
    """W [n_p, ng] and the pair energies [n, n] of the pairs (i occupied, j)."""
    shape, dv = _shape(case), _dv(case)
    k = _k_table(case, psi.device)
    W = torch.zeros_like(psi)
    e = torch.zeros((n, n), dtype=torch.float64, device=psi.device)
    per = max(1, (1 << 26) // psi.shape[1])
    for at in range(0, len(pairs), per):
        i, j = pairs[at:at + per, 0], pairs[at:at + per, 1]
        rho = psi[i] * psi[j]
        v = torch.fft.irfftn(torch.fft.rfftn(rho.view(-1, *shape), dim=(1, 2, 3)) * k, s=shape, dim=(1, 2, 3)).reshape(rho.shape)
        W.index_add_(0, j, -psi[i] * v)
        both = (j < n) & (i != j)
        W.index_add_(0, i[both], -psi[j[both]] * v[both])
        occ = j < n
        val = dv * (rho[occ] * v[occ]).sum(1)
        e[i[occ], j[occ]] = val
        e[j[occ], i[occ]] = val
    return W, e


def _exact_step(case, seed):
    n, p, dv, shape = case["n_occ"], case["n_occ"] + case["n_extra"], _dv(case), _shape(case)
    phi, trial = _inputs(case, seed)
    phi = phi.view(p, -1)
    occ = _lowdin(phi[:n], dv)
    if case["kind"] == "plain":
        idx = torch.triu_indices(n, n, device=phi.device).T
        W, e = _exchange(case, occ, n, idx)
        return {"W": W.view((n,) + shape), "ex": -0.5 * float(e.sum())}
    sub = occ.view((n,) + shape)[:, ::2, ::2, ::2]
    m = sub.shape[1:]
    r = sub.reshape(n, -1).clone()
    picked = []
    for _ in range(n):
        at = int(torch.argmax((r * r).sum(0)))
        picked.append(at)
        q = r[:, at] / torch.linalg.norm(r[:, at])
        r -= torch.outer(q, q @ r)
    pc = torch.tensor(picked, device=phi.device)
    full = ((pc // (m[1] * m[2]) * 2) * shape[1] + (pc // m[2]) % m[1] * 2) * shape[2] + pc % m[2] * 2
    c = occ[:, full].T  # points x orbitals
    w = (c.T @ _inv_sqrt(c @ c.T)).T @ occ
    psi = w
    if case["n_extra"]:
        x = phi[n:] - (dv * (phi[n:] @ occ.T)) @ occ
        psi = torch.cat([w, _lowdin(x, dv)])
    del phi, occ, r, sub
    s = torch.zeros((n, n), dtype=torch.float64, device=w.device)
    for at in range(0, w.shape[1], 1 << 18):
        a = w[:, at:at + (1 << 18)].abs()
        s += dv * (a @ a.T)
    keep = torch.triu(s >= S_THR)
    pairs = torch.nonzero(keep)
    if case["n_extra"]:
        i = torch.arange(n, device=w.device).repeat_interleave(case["n_extra"])
        j = torch.arange(n, p, device=w.device).repeat(n)
        pairs = torch.cat([pairs, torch.stack([i, j], 1)])
    W, e = _exchange(case, psi, n, pairs)
    out = {"n_pairs": None, "ex": -0.5 * float(e.sum()), "e": e}
    if trial is not None:
        M = dv * (psi @ W.T)
        L = torch.linalg.cholesky(-0.5 * (M + M.T))
        xi = torch.linalg.solve_triangular(L, W, upper=False)
        X = dv * (trial.view(len(trial), -1) @ xi.T)
        out["kpsi"] = -(X @ xi).view((-1,) + shape)
        out["e_block"] = -float((X * X).sum())
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("serve", "batch"):
        got = [_exact_step(c, seed * 64 + k) for k, c in enumerate(_sub(case))]
        if kind == "batch":
            return {"ex": np.array([g["ex"] for g in got]), "pair_e": [g["e"] for g in got]}
        return {"%s%d" % (key, k): g[key] for k, g in enumerate(got) for key in ("ex", "kpsi")}
    got = _exact_step(case, seed)
    if kind == "plain":
        return got
    if kind == "apply":
        return {"kpsi": got["kpsi"], "e_block": got["e_block"]}
    return {"n_pairs": None, "ex": got["ex"], "kpsi": got["kpsi"]}
