"""The work a user of this framework has it do, as cases that can be timed and compared.

Each case goes through the public entry points of ``paper_2110_03607_gb300``: whole runs from
the Ising tensor, one coarse-graining step of a tensor that the program holds (a resume, or
one step of a scan), its layers (the environment Grams, the contraction of a rank's share of
the slices, the bottleneck product alone), a batch of independent steps, and the derivative of
ln Z with respect to beta through torch.autograd.  ``exact`` restates each in plain torch in
64 bits.

The tensors are those of a block of Ising spins with random ferromagnetic couplings: a leg of
bond dimension chi bundles ceil(log2 chi) bonds that leave the block and keeps its chi leading
channels.  They have the parity blocks of the spin-flip symmetry at zero field and the decay
along every leg that coarse-grained Ising tensors have, and no accidental degeneracy, so that
the kept eigenvectors are the same for every correct solver.
"""

import math

import numpy as np
import torch

import paper_2110_03607_gb300 as hotrg

FORMS = {"fp64": hotrg.PREC_FP64, "bf16x3": hotrg.PREC_BF16X3, "bf16x6": hotrg.PREC_BF16X6,
         "tf32x3": hotrg.PREC_TF32X3}
FP64_BELOW = 2.0 ** 36   # the default bottleneck size below which a step is contracted in FP64


def _step(name, c, axis, chi, field, form):
    k = list(c) + [0] * (4 - len(c))
    case = {"kind": "step", "d": len(c), "c0": k[0], "c1": k[1], "c2": k[2], "c3": k[3], "axis": axis,
            "chi": chi, "field": field, "form": form}
    return dict(case, name=name) if name else case


def listed():
    return [
        # a whole run from the Ising tensor, as a first-time user or a test makes it: every step
        # is small and the time is launches and latency
        {"name": "run2d_chi8", "kind": "run", "d": 2, "chi": 8, "h": 0.0, "steps": 12},
        # a 2D step at the bond dimension of a production 2D run: the eigen-solver is the work
        _step("step2d_chi24", (24, 24), 1, 24, 0.0, "bf16x6"),
        # the headline workload: one 3D step at zero field (Z2 blocks, split BF16)
        _step("step3d_chi16", (16, 16, 16), 2, 16, 0.0, "bf16x6"),
        # the largest 3D run: bond dimension 20
        _step("step3d_chi20", (20, 20, 20), 0, 20, 0.0, "bf16x6"),
        # a magnetisation scan: a field breaks the spin-flip symmetry, every step is dense
        _step("field3d_chi12", (12, 12, 12), 1, 12, 0.02, "bf16x6"),
        # a step in plain FP64 with unequal bonds, as references and early steps are made
        _step("fp64_3d_ragged", (9, 11, 10), 0, 11, 0.01, "fp64"),
        # 4D at zero field
        _step("step4d_chi6", (6, 6, 6, 6), 3, 6, 0.0, "bf16x6"),
        # the energy from ln Z: forward with the derivative carried, and the backward pass
        {"name": "energy2d_chi12", "kind": "energy", "d": 2, "chi": 12, "h": 0.02, "steps": 8, "order": 1},
        # a scan over beta and h: independent instances stepped together
        {"name": "batch3d", "kind": "batch", "n": 8, "lo": 6, "hi": 12, "form": "bf16x6"},
        # the bottleneck product on its own, odd sizes, for a caller that owns its memory
        {"name": "gemm_ragged", "kind": "gemm", "m": 1001, "n": 1500, "k": 1333, "form": "bf16x6"},
        # the environment Grams of a 3D step (one rank's share of one)
        {"name": "env3d_chi16", "kind": "env", "d": 3, "c0": 16, "c1": 16, "c2": 16, "c3": 0, "axis": 0,
         "chi": 16, "field": 0.0},
        # the contraction of a rank's slices in a dense step, split TF32
        {"name": "contract3d_chi13", "kind": "contract", "d": 3, "c0": 13, "c1": 13, "c2": 13, "c3": 0,
         "axis": 0, "chi": 13, "field": 0.02, "form": "tf32x3", "slices": 4},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choice(["run", "step", "step", "step", "step", "energy", "batch", "gemm", "env", "contract"])
    if kind == "run":
        return {"kind": "run", "d": 2, "chi": rng.randint(4, 16), "h": rng.choice([0.0, 0.05]),
                "steps": rng.randint(4, 16)}
    if kind == "energy":
        if rng.random() < 0.5:
            return {"kind": "energy", "d": 2, "chi": rng.randint(6, 14), "h": rng.choice([0.02, 0.05]),
                    "steps": rng.randint(4, 8), "order": rng.choice([1, 2])}
        return {"kind": "energy", "d": 2, "chi": rng.randint(6, 12), "h": rng.choice([0.01, 0.1]),
                "steps": rng.randint(5, 9), "order": 1}
    if kind == "batch":
        return {"kind": "batch", "n": rng.randint(2, 16), "lo": rng.randint(5, 7), "hi": rng.randint(9, 12),
                "form": rng.choice(["bf16x6", "tf32x3", "bf16x3"])}
    if kind == "gemm":
        form = rng.choice(["bf16x6", "bf16x3", "fp64"])
        return {"kind": "gemm", "m": _log_int(rng, 33, 1800), "n": _log_int(rng, 33, 1800),
                "k": _log_int(rng, 17, 1800), "form": form}
    d = rng.choice([2, 3, 3, 4])
    field = rng.choice([0.0, 0.0, 0.02])
    form = rng.choice(["bf16x6", "bf16x6", "tf32x3", "bf16x3", "fp64"])
    if kind == "contract" and d == 2:
        d = 3
    if d == 2:
        c = [rng.randint(6, 28)] * 2
    elif d == 3:
        top = 11 if form == "fp64" else (14 if field else 18)
        base = _log_int(rng, 5, top)
        c = [max(2, min(top, base + rng.choice([0, 0, 0, -1, 1]))) for _ in range(3)]
    else:
        top = 5 if form == "fp64" else 6
        base = rng.randint(3, top)
        c = [max(2, min(top, base + rng.choice([0, 0, -1]))) for _ in range(4)]
    axis = rng.randrange(d)
    chi = max(c)
    case = _step(None, c, axis, chi, field, form)
    if kind == "env":
        del case["form"]
        return dict(case, kind="env")
    if kind == "contract":
        return dict(case, kind="contract", slices=rng.randint(1, min(4, c[axis])))
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
SPINS = 8   # of a block: 2 x 2 x 2 in 3D


def _chis(case):
    return [case["c%d" % k] for k in range(case["d"])]


def _block_tensor(chis, field, seed, dev):
    """(tensor in the interchange layout (x_1, x_1', x_2, x_2', ..), trace 1; parity of every index)."""
    rng = np.random.default_rng(seed)
    d = len(chis)
    beta = {2: 0.38, 3: 0.24, 4: 0.20}[d] * rng.uniform(0.97, 1.03)
    ncfg = 1 << SPINS
    sig = 1.0 - 2.0 * ((np.arange(ncfg)[:, None] >> np.arange(SPINS)[None, :]) & 1)
    logw = beta * field * sig.sum(1)
    for a in range(SPINS):          # the bonds of a cube
        for bit in range(3):
            b = a ^ (1 << bit)
            if b > a:
                logw += beta * rng.uniform(0.6, 1.4) * sig[:, a] * sig[:, b]
    w = np.exp(logw - logw.max())
    fac, par = [], []
    for c in chis:
        nb = max(1, math.ceil(math.log2(c)))
        both = [(rng.permutation(SPINS)[:nb], beta * rng.uniform(0.6, 1.4, nb)) for _ in range(2)]
        idx = np.arange(1 << nb)
        bits = (idx[:, None] >> np.arange(nb)[None, :]) & 1
        lead = (bits * 0.5 * np.log(np.tanh(both[0][1]) * np.tanh(both[1][1]))[None, :]).sum(1)
        keep = np.argsort(-lead, kind="stable")[:c]
        par.append((bits[keep].sum(1) & 1).astype(int))
        legs = []
        for sites, bj in both:
            f = np.ones((ncfg, c))
            for q in range(nb):
                x0, x1 = math.sqrt(math.cosh(bj[q])), math.sqrt(math.sinh(bj[q]))
                f = f * np.where(bits[keep, q][None, :] == 1, sig[:, sites[q]][:, None] * x1, x0)
            legs.append(f)
        fac.append(legs)

    def rows(side):
        m = torch.ones(ncfg, 1, dtype=torch.float64, device=dev)
        for k in range(d):
            f = torch.tensor(fac[k][side], dtype=torch.float64, device=dev)
            m = (m[:, :, None] * f[:, None, :]).reshape(ncfg, -1)
        return m

    r, cpr = rows(0), rows(1)
    t = (r * torch.tensor(w, dtype=torch.float64, device=dev)[:, None]).T @ cpr
    if field == 0.0:   # the sum over spin flips cancels exactly on odd total parity
        pr = np.zeros(1, dtype=int)
        for k in range(d):
            pr = (pr[:, None] ^ par[k][None, :]).reshape(-1)
        pt = torch.tensor(pr, device=dev)
        t = torch.where(pt[:, None] == pt[None, :], t, torch.zeros((), dtype=t.dtype, device=dev))
    t = t / torch.trace(t)
    perm = [v for k in range(d) for v in (k, d + k)]
    return t.reshape(list(chis) * 2).permute(perm).contiguous(), par


def _field_or_parity(case, par):
    return [int(v) for p in par for v in p] if case["field"] == 0.0 else None


def _is_fp64(case, chis, axis, chi):
    """Whether the step's contraction runs in FP64 (the form asked for, or a small bottleneck)."""
    return case["form"] == "fp64" or _bottleneck(chis, axis, chi) < FP64_BELOW


def _beta_of(seed):
    return float(np.random.default_rng(seed).uniform(0.40, 0.46))


def _context(case, chis, tensor, parity):
    g = hotrg.Hotrg(len(chis), 0.25, case["field"], precision=FORMS[case.get("form", "bf16x6")], tensor=tensor,
                    chis=chis)
    if parity is not None:
        hotrg.hotrg_set_parity(g.ctx, parity)
    return g


def _out_shape(chis, axis, chi):
    return [chis[k] if k == axis else min(chis[k] ** 2, chi) for k in range(len(chis)) for _ in range(2)]


def prepare(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    if kind in ("run", "energy"):
        return {"case": case, "beta": _beta_of(seed)}
    if kind == "gemm":
        gen = torch.Generator(device=dev).manual_seed(seed)
        # rows of a coarse-grained tensor fall off along every leg
        fall = torch.exp(-1.5 * torch.rand(case["k"], generator=gen, device=dev, dtype=torch.float64))
        a, b = [torch.randn(r, case["k"], generator=gen, device=dev, dtype=torch.float64) * fall
                for r in (case["m"], case["n"])]
        return {"case": case, "a": a, "b": b, "c": torch.empty(case["m"], case["n"], dtype=torch.float64, device=dev)}
    if kind == "batch":
        items = []
        for one, s in _instances(case, seed):
            t, par = _block_tensor(_chis(one), one["field"], s, dev)
            items.append((_context(one, _chis(one), t, _field_or_parity(one, par)), one, t, _field_or_parity(one, par),
                          torch.empty(_out_shape(_chis(one), one["axis"], one["chi"]), dtype=torch.float64, device=dev),
                          torch.cuda.Stream()))
        for g, _, _, _, _, st in items:
            hotrg.hotrg_set_stream(g.ctx, st.cuda_stream)
        return {"case": case, "items": items}
    chis = _chis(case)
    t, par = _block_tensor(chis, case["field"], seed, dev)
    parity = _field_or_parity(case, par)
    state = {"case": case, "chis": chis, "t": t, "parity": parity, "g": _context(case, chis, t, parity)}
    if kind == "step":
        state["out"] = torch.empty(_out_shape(chis, case["axis"], case["chi"]), dtype=torch.float64, device=dev)
    else:
        ctx = state["g"].ctx
        grams, _, per = hotrg.shard_sizes(ctx, case["axis"], case["chi"])
        state["grams"] = torch.empty(grams, dtype=torch.float64, device=dev)
        if kind == "contract":
            hotrg.hotrg_shard_env(ctx, case["axis"], case["chi"], 0, 1, out=state["grams"])
            hotrg.hotrg_shard_isometries(ctx, case["axis"], case["chi"], state["grams"])
            state["slices"] = torch.empty(case["slices"] * per, dtype=torch.float64, device=dev)
    return state


def _instances(case, seed):
    """The batch's instances: bond dimensions lo .. hi, every other one with a field."""
    for i in range(case["n"]):
        c = case["lo"] + (case["hi"] - case["lo"]) * (i // 2) // max(1, (case["n"] - 1) // 2)
        one = _step(None, (c, c, c), i % 3, c, 0.0 if i % 2 == 0 else 0.01, case["form"])
        yield one, seed * 64 + i


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _load(ctx, chis, tensor, parity):
    """What a program does to step a tensor that it holds (a checkpoint, one point of a scan)."""
    hotrg.hotrg_set_tensor(ctx, chis, tensor)
    if parity is not None:
        hotrg.hotrg_set_parity(ctx, parity)


def _kept(out, fp64):
    """The new tensor as the program keeps it: the split forms sum in FP32, so FP32 holds all of it."""
    return out if fp64 else out.float()


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "run":
        g = hotrg.Hotrg(case["d"], state["beta"], case["h"])
        for i in range(case["steps"]):
            g.step(i % case["d"], case["chi"])
        lnz, _ = g.free_energy()
        trace, x, _ = hotrg.hotrg_observables(g.ctx)
        leg = case["steps"] % case["d"]   # a leg across the last step's axis
        spectra = [hotrg.hotrg_spectrum(g.ctx, leg, prime) for prime in (0, 1)]
        g.close()
        return {"lnz": np.array([lnz]), "trace": trace, "x": x, "spectra": spectra}
    if kind == "energy":
        from paper_2110_03607_gb300 import autograd as ad

        beta = torch.tensor(state["beta"], dtype=torch.float64, requires_grad=True)
        axes = [i % case["d"] for i in range(case["steps"])]
        lnz = ad.ln_z_per_site(beta, case["d"], case["h"], case["chi"], axes, hotrg.PREC_FP64, case["order"])
        (grad,) = torch.autograd.grad(lnz[-1], beta, create_graph=case["order"] == 2)
        out = {"lnz": lnz.detach(), "grad": grad.detach()}
        if case["order"] == 2:
            (out["grad2"],) = torch.autograd.grad(grad, beta)
        return out
    if kind == "gemm":
        hotrg.hotrg_gemm_nt_noalloc(FORMS[case["form"]], state["a"], state["b"], state["c"],
                                    torch.cuda.current_stream().cuda_stream)
        return _kept(state["c"], case["form"] == "fp64")
    if kind == "batch":
        items = state["items"]
        for g, one, t, parity, _, _ in items:
            _load(g.ctx, _chis(one), t, parity)
        hotrg.hotrg_step_batch([it[0].ctx for it in items], [it[1]["axis"] for it in items],
                               [it[1]["chi"] for it in items])
        outs = []
        for g, one, _, _, out, _ in items:
            hotrg.hotrg_tensor(g.ctx, out=out)
            outs.append(_kept(out, _is_fp64(one, _chis(one), one["axis"], one["chi"])))
        return outs
    ctx, chis, axis, chi = state["g"].ctx, state["chis"], case["axis"], case["chi"]
    if kind == "env":
        _load(ctx, chis, state["t"], state["parity"])
        return hotrg.hotrg_shard_env(ctx, axis, chi, 0, 1, out=state["grams"])
    if kind == "contract":
        hotrg.hotrg_shard_contract(ctx, axis, chi, 0, case["slices"], out=state["slices"])
        return _kept(state["slices"], _is_fp64(case, chis, axis, chi))
    _load(ctx, chis, state["t"], state["parity"])
    hotrg.hotrg_step(ctx, axis, chi)
    hotrg.hotrg_tensor(ctx, out=state["out"])
    trace, x, _ = hotrg.hotrg_observables(ctx)
    spectra = [hotrg.hotrg_spectrum(ctx, leg, prime) for leg in range(case["d"]) if leg != axis for prime in (0, 1)]
    return {"tensor": _kept(state["out"], _is_fp64(case, chis, axis, chi)), "trace": trace, "x": x, "spectra": spectra}


# ---------------------------------------------------------------------------
# the work of a pass
# ---------------------------------------------------------------------------
def _bottleneck(chis, axis, chi):
    """Flops of the dense bottleneck: 2 R^2 (P_new P) per slice."""
    r = math.prod(chis)
    p = r // chis[axis]
    pn = math.prod(min(c * c, chi) for k, c in enumerate(chis) if k != axis)
    return 2.0 * r * r * pn * p * chis[axis]


def _gram_flops(chis, axis):
    """Flops of the symmetric products of the four Grams of every transverse leg."""
    rr = float(math.prod(chis)) ** 2
    return sum(4.0 * rr * (c * chis[axis] + 1) for k, c in enumerate(chis) if k != axis)


def _step_work(chis, axis, chi, z2, slices=None):
    r = math.prod(chis)
    rn = chis[axis] * math.prod(min(c * c, chi) for k, c in enumerate(chis) if k != axis)
    share = 1.0 if slices is None else slices / chis[axis]
    flops = _bottleneck(chis, axis, chi) * share / (4.0 if z2 else 1.0)
    if slices is None:
        flops += _gram_flops(chis, axis) / (4.0 if z2 else 1.0)
    return {"bytes": 8.0 * (r * r + rn * rn * share), "flops": flops}


def work(case):
    kind = case["kind"]
    if kind in ("run", "energy"):
        c, total = [2] * case["d"], {"bytes": 0.0, "flops": 0.0}
        for i in range(case["steps"]):
            w = _step_work(c, i % case["d"], case["chi"], kind == "run" and case["h"] == 0.0)
            total = {k: total[k] + w[k] * (1 if kind == "run" else 1 + 2 * case["order"]) for k in w}
            c = [v if k == i % case["d"] else min(v * v, case["chi"]) for k, v in enumerate(c)]
        return total
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 8.0 * (m * k + n * k + m * n), "flops": 2.0 * m * n * k}
    if kind == "batch":
        ws = [_step_work(_chis(o), o["axis"], o["chi"], o["field"] == 0.0) for o, _ in _instances(case, 0)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    chis, axis, z2 = _chis(case), case["axis"], case["field"] == 0.0
    if kind == "env":
        r = math.prod(chis)
        out = sum(4 * (c * chis[axis]) ** 2 for k, c in enumerate(chis) if k != axis)
        return {"bytes": 8.0 * (r * r + out), "flops": _gram_flops(chis, axis) / (4.0 if z2 else 1.0)}
    return _step_work(chis, axis, case["chi"], z2, case.get("slices") if kind == "contract" else None)


# ---------------------------------------------------------------------------
# 64 bits
# ---------------------------------------------------------------------------
def _slots(t, chis, axis):
    """The tensor as [c, n_1 .. | c', n_1' ..] and its bond dimensions in that order."""
    d = len(chis)
    to = [(axis + k) % d for k in range(d)]
    return t.permute([2 * v for v in to] + [2 * v + 1 for v in to]).contiguous(), [chis[v] for v in to], to


def _grams(ts, j):
    """S^ (free n_j, c'), S~ (n_j, c), S^' (n_j', c'), S~' (n_j', c)."""
    d = ts.ndim // 2
    out = []
    for f, cur in ((j, d), (j, 0), (d + j, d), (d + j, 0)):
        x = ts.permute([f, cur] + [q for q in range(2 * d) if q not in (f, cur)])
        x = x.reshape(x.shape[0] * x.shape[1], -1)
        out.append(x @ x.T)
    return out


def _eig(a, par):
    """Eigenvalues descending and their vectors (columns); by parity blocks where they are known."""
    n = a.shape[0]
    sets = [torch.arange(n, device=a.device)] if par is None else [torch.nonzero(par == b).flatten() for b in (0, 1)]
    lam, vec = [], []
    for rows in sets:
        if rows.numel():
            e, v = torch.linalg.eigh(a[rows][:, rows])
            full = torch.zeros(n, rows.numel(), dtype=a.dtype, device=a.device)
            full[rows] = v
            lam.append(e)
            vec.append(full)
    lam, vec = torch.cat(lam).abs(), torch.cat(vec, 1)
    order = torch.argsort(lam, descending=True)
    return lam[order], vec[:, order]


def _isometry(s_hat, s_chk, chi_j, chi_c, par):
    sh = s_hat.reshape(chi_j, chi_c, chi_j, chi_c).permute(0, 2, 1, 3).reshape(chi_j * chi_j, -1)
    sc = s_chk.reshape(chi_j, chi_c, chi_j, chi_c).permute(0, 2, 1, 3).reshape(chi_j * chi_j, -1)
    a = (sh @ sc.T).reshape(chi_j, chi_j, chi_j, chi_j)            # [f^, g^, f~, g~]
    a = a.permute(2, 0, 3, 1).reshape(chi_j * chi_j, chi_j * chi_j)  # row f^ + f~ chi_j
    return _eig(0.5 * (a + a.T), par)


def _isometries(ts, sizes, chi, pars):
    """Per transverse leg: the kept, sign-fixed U and the spectra of both sides."""
    d = len(sizes)
    us, spectra = [], []
    for j in range(1, d):
        par = None
        if pars is not None:
            par = (pars[j][:, None] ^ pars[j][None, :]).reshape(-1)
        s = _grams(ts, j)
        lam, v = _isometry(s[0], s[1], sizes[j], sizes[0], par)
        lamp, vp = _isometry(s[2], s[3], sizes[j], sizes[0], par)
        keep = min(sizes[j] ** 2, chi)
        prime = not (lam[keep:].sum() < lamp[keep:].sum() - 1e-10 * max(lam[0], lamp[0]))
        u = (vp if prime else v)[:, :keep]
        big = u.abs().max(0).values
        pivot = (u.abs() >= (1 - 1e-6) * big).double().argmax(0)
        u = u * torch.where(u.gather(0, pivot[None, :])[0] < 0, -1.0, 1.0)
        us.append(u)
        spectra.append((lam, lamp))
    return us, spectra


def _slice_of(ts, sizes, us, sl, row_par, new_par):
    """The c'-slice sl of the new tensor, [(c, n), n'] (unnormalised)."""
    d = len(sizes)
    r = math.prod(sizes)
    tm = ts.reshape(r, r)
    x = ts.select(d, sl)                                  # [rho, n~.. , n~'..]
    keep = [u.shape[1] for u in us]
    for j in range(1, d):                                 # n~'_j -> (n^'_j, n'_j), appended last
        u3 = us[j - 1].reshape(sizes[j], sizes[j], keep[j - 1])   # [check, hat, n']
        x = torch.tensordot(x, u3, dims=([d], [0]))
    m = d - 1                                             # [rho, n~ (m), (hat, n') x m]
    hats, news = [d + 2 * q for q in range(m)], [d + 2 * q + 1 for q in range(m)]
    x = x.permute(news + list(range(1, d)) + [0] + hats)
    b = x.reshape(-1, r)                                  # rows (n', n~), columns (rho, n^')
    if row_par is None:
        c = tm @ b.T
    else:
        pn = torch.zeros(1, dtype=torch.long, device=b.device)
        for p in new_par + row_par[1]:
            pn = (pn[:, None] ^ p[None, :]).reshape(-1)
        c = torch.zeros(r, b.shape[0], dtype=b.dtype, device=b.device)
        for par in (0, 1):
            rows = torch.nonzero(row_par[0] == par).flatten()
            cols = torch.nonzero(pn == (par ^ row_par[2][sl])).flatten()
            if rows.numel() and cols.numel():
                c[rows[:, None], cols[None, :]] = tm[rows][:, rows] @ b[cols][:, rows].T
    c = c.reshape(list(sizes) + keep + list(sizes[1:]))   # [c, n^.., n'.., n~..]
    for j in range(m, 0, -1):                             # (n^_j, n~_j) -> n_j, appended last
        u3 = us[j - 1].reshape(sizes[j], sizes[j], keep[j - 1])   # [check, hat, n]
        c = torch.tensordot(c, u3, dims=([j, 2 * j + m], [1, 0]))
        # the n_j appended so far stand last, in the order m .. j; the axes before keep theirs
    # now [c, n'.. (m), n_m .. n_1]
    c = c.permute([0] + [1 + m + (m - 1 - q) for q in range(m)] + list(range(1, 1 + m)))
    return c.reshape(sizes[0] * math.prod(keep), math.prod(keep))


def _exact_step(t, chis, axis, chi, par, slices=None):
    """(new tensor in the interchange layout normalised by its trace, trace, X, spectra by lattice
    axis, new parities), or the first `slices` c'-slices as the shard lays them out."""
    ts, sizes, to = _slots(t, chis, axis)
    d = len(chis)
    pars = None if par is None else [torch.tensor(par[v], device=t.device) for v in to]
    us, spectra = _isometries(ts, sizes, chi, pars)
    keep = [u.shape[1] for u in us]
    row_par = new_par = None
    if pars is not None:
        rp = torch.zeros(1, dtype=torch.long, device=t.device)
        for p in pars:
            rp = (rp[:, None] ^ p[None, :]).reshape(-1)
        row_par = (rp, pars[1:], [int(v) for v in pars[0]])
        new_par = []
        for j, u in enumerate(us):
            comp = (pars[j + 1][:, None] ^ pars[j + 1][None, :]).reshape(-1)
            new_par.append(comp[u.abs().argmax(0)])
    n = sizes[0] if slices is None else slices
    parts = [_slice_of(ts, sizes, us, sl, row_par, new_par) for sl in range(n)]
    if slices is not None:
        return torch.stack(parts)
    tn = torch.stack(parts, 1).reshape([sizes[0]] + keep + [sizes[0]] + keep)   # [c, n.., c', n'..]
    pn = math.prod(keep)
    y = torch.einsum("anbn->ab", tn.reshape(sizes[0], pn, sizes[0], pn))
    trace = torch.trace(y)
    x = trace * trace / (y * y.T).sum()
    tn = tn / trace
    back = [to.index(k) for k in range(d)]
    tn = tn.permute([v for k in back for v in (k, d + k)]).contiguous()
    out_par = None
    if pars is not None:
        out_par = [None] * d
        out_par[to[0]] = np.asarray(par[to[0]])
        for j in range(1, d):
            out_par[to[j]] = new_par[j - 1].cpu().numpy()
    by_axis = [spectra[to.index(k) - 1] for k in range(d) if k != axis]
    return tn, float(trace), float(x), [s.cpu().numpy() for pair in by_axis for s in pair], out_par


def _exact_run(case, beta):
    """ln Z / V after every step, and the last step's trace, X and spectra, from the Ising tensor."""
    d, h = case["d"], case["h"]
    x = np.array([[math.sqrt(math.cosh(beta)), math.sqrt(math.sinh(beta))],
                  [math.sqrt(math.cosh(beta)), -math.sqrt(math.sinh(beta))]])
    t = np.zeros([2] * (2 * d))
    for s, sg in ((0, 1.0), (1, -1.0)):
        f = np.array(math.exp(beta * h * sg))
        for _ in range(2 * d):
            f = f[..., None] * x[s]
        t = t + f
    t = torch.tensor(t)
    tr = float(torch.einsum("aabb->" if d == 2 else "aabbcc->", t)) if d < 4 else float(torch.einsum("aabbccdd->", t))
    par = [np.array([0, 1])] * d if h == 0.0 else None
    t, chis, kappa, ln_tr, rows = t / tr, [2] * d, 0.0, math.log(tr), []
    for i in range(case["steps"]):
        t, trace, gw, spectra, par = _exact_step(t, chis, i % d, case["chi"], par)
        chis = list(t.shape[0::2])
        kappa += ln_tr / 2.0 ** i
        ln_tr = math.log(trace)
        rows.append(kappa + ln_tr / 2.0 ** (i + 1))
    return rows, trace, gw, spectra


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    kind = case["kind"]
    if kind == "run":
        rows, trace, x, spectra = _exact_run(case, _beta_of(seed))
        return {"lnz": np.array(rows[-1:]), "trace": trace, "x": x, "spectra": spectra[:2]}
    if kind == "energy":
        rows, _, _, _ = _exact_run(case, _beta_of(seed))
        return {"lnz": torch.tensor(rows, dtype=torch.float64), "grad": None, **({"grad2": None} if case["order"] == 2 else {})}
    if kind == "gemm":
        s = prepare(case, seed)
        return s["a"] @ s["b"].T
    if kind == "batch":
        outs = []
        for one, s in _instances(case, seed):
            t, par = _block_tensor(_chis(one), one["field"], s, dev)
            outs.append(_exact_step(t, _chis(one), one["axis"], one["chi"], par if one["field"] == 0.0 else None)[0])
        return outs
    chis, axis, chi = _chis(case), case["axis"], case["chi"]
    z2 = case["field"] == 0.0
    if _step_work(chis, axis, chi, z2, case.get("slices") if kind == "contract" else None)["flops"] > 1.2e13:
        return None
    t, par = _block_tensor(chis, case["field"], seed, dev)
    if kind == "env":
        ts, sizes, _ = _slots(t, chis, axis)
        return torch.cat([s.reshape(-1) for j in range(1, case["d"]) for s in _grams(ts, j)])
    got = _exact_step(t, chis, axis, chi, par if z2 else None, case["slices"] if kind == "contract" else None)
    if kind == "contract":
        return got.reshape(-1)
    return {"tensor": got[0], "trace": got[1], "x": got[2], "spectra": got[3]}
