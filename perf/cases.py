"""Workloads of the equalizer library, as its users call it: one pass each, on the GPU.

Four kinds of pass:

* ``equalize``  ``ffeq_equalize`` on a kept plan, workspace and output buffers: PD or FD; L-MMSE, ZF,
                MRC or LAMA; every precision; with or without refinement; soft outputs.
* ``uneven``    ``ffeq_batch_equalize`` on a kept batch: instances of different sizes and noise levels.
* ``train``     a training step of the differentiable FD form with free regularizers and fusion
                weights: ``autograd.fd_equalize`` and its backward.
* ``optimal``   the same through the optimal fusion weights: ``autograd.fd_equalize_optimal``.

Inputs follow the uplink model y = H s + n: CN(0, 1) channels, optionally with exponential receive
correlation, square QAM of energy Es = 1, and N0 = U Es / SNR.  ``exact`` restates the equalizers in
64-bit torch, without the library's code.
"""
import math

import torch

from paper_1808_04473_gb300 import autograd, ffeq

ARCH = {"pd": ffeq.PD, "fd": ffeq.FD}
PRECISION = {"fp32": ffeq.FP32, "tf32x3": ffeq.TF32X3, "bf16x3": ffeq.BF16X3, "fp16x3": ffeq.FP16X3}
EQUALIZER = {"lmmse": ffeq.LMMSE, "zf": ffeq.ZF, "mrc": ffeq.MRC, "lama": ffeq.LAMA}
ES = 1.0


def _equalize(name=None, **kw):
    c = dict(kind="equalize", arch="fd", precision="fp32", equalizer="lmmse", B=256, U=16, C=8, n_sc=1200, n_sym=14,
             bits=4, snr_db=10.0, corr=0.0, refine=0, refine_fp64=0, iters=0, info=False)
    c.update(kw)
    return {**({"name": name} if name else {}), **c}


def listed():
    return [
        # The smallest call in use: one short pilot block, 64 subcarriers of one symbol; latency of the launches.
        _equalize("fd_small_fp32", B=32, U=4, C=2, n_sc=64, n_sym=1, bits=2, info=True),
        # One OFDM slot of the large array at the tensor-core precision, both architectures.
        _equalize("pd_slot_bf16x3", arch="pd", precision="bf16x3"),
        _equalize("fd_slot_bf16x3", precision="bf16x3"),
        # The same slot at the library's default precision.
        _equalize("fd_slot_fp32"),
        # A wide-band slot over correlated channels with clusters smaller than the number of users.
        _equalize("fd_wide_corr_fp16x3", precision="fp16x3", U=32, C=16, n_sc=3300, bits=6, snr_db=15.0, corr=0.7),
        # The same, refined from the inputs, the residual in FP64 where the system is ill-conditioned.
        _equalize("fd_wide_corr_refined", precision="fp16x3", U=32, C=16, n_sc=3300, bits=6, snr_db=15.0, corr=0.7,
                  refine=1, refine_fp64=1),
        # The nonlinear equalizer on the slot.
        _equalize("fd_slot_lama", precision="bf16x3", equalizer="lama", iters=8),
        # Sizes that fill no tile: 12 users on 100 antennas, zero forcing at TF32x3.
        _equalize("pd_ragged_zf_tf32x3", arch="pd", precision="tf32x3", equalizer="zf", B=100, U=12, C=5, n_sc=333,
                  n_sym=7, snr_db=15.0, info=True),
        # 11 users on clusters of 24 antennas.
        _equalize("fd_ragged_bf16x3", precision="bf16x3", B=120, U=11, C=5, n_sc=625, n_sym=13, bits=6),
        # Many cells served in one call, each with its own sizes and noise.
        dict(name="fd_uneven_bf16x3", kind="uneven", arch="fd", precision="bf16x3", equalizer="lmmse", n_inst=4096,
             U_min=4, U_max=32, sym_max=14, bits=4, sizes_seed=77),
        # Training steps: 8 channel draws of 1024 subcarriers, forward and backward.
        dict(name="train_free_weights", kind="train", B=128, U=16, C=8, n_sc=8192, n_sym=1, bits=2, snr_db=10.0),
        dict(name="train_optimal_weights", kind="optimal", B=128, U=16, C=8, n_sc=8192, n_sym=1, bits=2, snr_db=10.0),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["equalize", "equalize", "equalize", "equalize", "uneven", "train", "optimal"])
    if kind == "uneven":
        lo = rng.randint(1, 8)
        return dict(kind="uneven", arch=rng.choice(["pd", "fd"]), precision=rng.choice(["fp32", "tf32x3", "bf16x3"]),
                    equalizer=rng.choice(["lmmse", "lmmse", "mrc"]), n_inst=_log_int(rng, 64, 4096), U_min=lo,
                    U_max=rng.randint(max(lo, 8), 32), sym_max=rng.randint(1, 14), bits=rng.choice([2, 4, 6]),
                    sizes_seed=rng.randint(1, 10 ** 6))
    if kind in ("train", "optimal"):
        U = rng.randint(2, 16)
        C = rng.choice([1, 2, 3, 4, 5, 8])
        S = rng.randint(4, 128 // C)
        n_sym = rng.choice([1, 1, 2, 3, 6])
        return dict(kind=kind, B=S * C, U=U, C=C, n_sc=_log_int(rng, 64, 8192 // n_sym), n_sym=n_sym,
                    bits=rng.choice([2, 4]), snr_db=round(rng.uniform(0.0, 15.0), 1))
    equalizer = rng.choice(["lmmse", "lmmse", "lmmse", "zf", "mrc", "lama"])
    arch = rng.choice(["pd", "fd"])
    precision = rng.choice(["fp32", "tf32x3", "bf16x3", "fp16x3"])
    U = rng.choice([rng.randint(1, 32), 4, 8, 16, 32])
    C = rng.choice([1, 2, 3, 4, 5, 8, 16])
    # LAMA and per-cluster zero forcing are used with at least twice as many antennas as users in a system, the
    # split precisions without refinement with at least as many.
    need = 2 * U if equalizer in ("lama", "zf") else (U if precision != "fp32" else 4)
    while C > 1 and need * (C if arch == "fd" else 1) > 256:
        C = C // 2
    S = rng.randint(max(1, -(-need // (1 if arch == "fd" else C))), 256 // C)
    refine = rng.choice([0, 0, 0, 1]) if equalizer in ("lmmse", "zf") else 0
    return _equalize(arch=arch, precision=precision, equalizer=equalizer, B=S * C, U=U, C=C,
                     n_sc=_log_int(rng, 64, 1200 if equalizer == "lama" else 3300), n_sym=rng.randint(1, 14),
                     bits=rng.choice([2, 4, 6, 8]) if equalizer != "lama" else rng.choice([2, 4]),
                     snr_db=round(rng.uniform(0.0, 18.0), 1), corr=rng.choice([0.0, 0.0, 0.5]), refine=refine,
                     refine_fp64=refine * rng.choice([0, 1]), iters=rng.randint(2, 8) if equalizer == "lama" else 0,
                     info=rng.choice([True, False]))


# ------------------------------------------------------------------------------------------- inputs

def _cn(shape, gen):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=gen, device="cuda") * math.sqrt(0.5))


def _symbols(shape, bits, gen):
    L = 1 << (bits // 2)
    lev = torch.randint(0, L, (*shape, 2), generator=gen, device="cuda").float() * 2 - (L - 1)
    return torch.view_as_complex(lev * math.sqrt(ES * 1.5 / (L * L - 1)))


def _n0(U, snr_db):
    return U * ES / 10.0 ** (snr_db / 10.0)


def _uplink(case, gen):
    """H [n_sc][U][B], y [n_sc][n_sym][B] and N0."""
    B, U, n_sc, n_sym = case["B"], case["U"], case["n_sc"], case["n_sym"]
    H = _cn((n_sc, U, B), gen)
    if case.get("corr"):
        i = torch.arange(B, device="cuda", dtype=torch.float64)
        R = case["corr"] ** (i[:, None] - i[None, :]).abs()
        H = torch.view_as_complex(torch.stack(
            [torch.matmul(p, torch.linalg.cholesky(R).float().T) for p in (H.real, H.imag)], dim=-1))
    N0 = _n0(U, case["snr_db"])
    y = torch.matmul(_symbols((n_sc, n_sym, U), case["bits"], gen), H) + math.sqrt(N0) * _cn((n_sc, n_sym, B), gen)
    return H.contiguous(), y.contiguous(), N0


def _uneven_specs(case):
    """Sizes and noise of every instance (B, U, C, n_sc, n_sym, N0, Es): part of the case, not of the seed."""
    g = torch.Generator().manual_seed(case["sizes_seed"])

    def integer(lo, hi):
        return int(torch.randint(lo, hi + 1, (), generator=g))

    specs = []
    for _ in range(case["n_inst"]):
        U, B = integer(case["U_min"], case["U_max"]), (64, 128, 256)[integer(0, 2)]
        Cs = [c for c in (1, 2, 4, 8, 16) if B // c >= 4]
        C, n_sym = Cs[integer(0, len(Cs) - 1)], integer(1, case["sym_max"])
        specs.append((B, U, C, 1, n_sym, _n0(U, 5.0 + 15.0 * float(torch.rand((), generator=g))), ES))
    return specs


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dev = "cuda"
    if case["kind"] == "equalize":
        B, U, C, n_sc, n_sym, bits = (case[k] for k in ("B", "U", "C", "n_sc", "n_sym", "bits"))
        H, y, N0 = _uplink(case, gen)
        plan = ffeq.ffeq_plan_create(B, U, C, n_sc, n_sym, arch=ARCH[case["arch"]], precision=PRECISION[case["precision"]],
                                     llr_bits=bits, refine=case["refine"], refine_fp64=case["refine_fp64"],
                                     equalizer=EQUALIZER[case["equalizer"]], lama_iters=case["iters"])
        nb = ffeq.ffeq_workspace_size(plan)
        s2 = (n_sc, n_sym, U) if case["equalizer"] == "lama" else (n_sc, U)
        out = dict(z=torch.empty((n_sc, n_sym, U), dtype=torch.complex64, device=dev),
                   sigma2=torch.empty(s2, device=dev), llr=torch.empty((n_sc, n_sym, U, bits), device=dev))
        if case["info"]:
            out["info"] = torch.empty((n_sc, C if case["arch"] == "fd" else 1), dtype=torch.int32, device=dev)
        return dict(case=case, plan=plan, H=H, y=y, N0=N0, out=out, nb=nb,
                    ws=torch.empty(max(nb, 16), dtype=torch.uint8, device=dev))
    if case["kind"] == "uneven":
        specs = _uneven_specs(case)
        cfg, inst = ffeq.pack_batch(specs, arch=ARCH[case["arch"]], precision=PRECISION[case["precision"]],
                                    llr_bits=case["bits"], equalizer=EQUALIZER[case["equalizer"]])
        batch = ffeq.ffeq_batch_create(cfg, inst)
        H, y = _cn((cfg.h_elems,), gen), _cn((cfg.y_elems,), gen)
        s = _symbols((sum(sp[1] * sp[4] for sp in specs),), case["bits"], gen)
        at = 0
        for sp, it in zip(specs, inst):
            B, U, n_sym = sp[0], sp[1], sp[4]
            yi = y[it.y_off:it.y_off + n_sym * B].view(n_sym, B)
            # y = s H + sqrt(N0) n, in place of the unit noise already there.
            torch.addmm(yi, s[at:at + n_sym * U].view(n_sym, U), H[it.h_off:it.h_off + U * B].view(U, B),
                        beta=math.sqrt(sp[5]), out=yi)
            at += n_sym * U
        out = dict(z=torch.zeros(cfg.z_elems, dtype=torch.complex64, device=dev),
                   sigma2=torch.zeros(cfg.sigma2_elems, device=dev), llr=torch.zeros(cfg.llr_elems, device=dev),
                   info=torch.zeros(cfg.info_elems, dtype=torch.int32, device=dev))
        nb = ffeq.ffeq_batch_workspace_size(batch)
        ws = torch.empty(nb, dtype=torch.uint8, device=dev)
        ffeq.ffeq_batch_upload(batch, ws, nb)
        return dict(case=case, batch=batch, specs=specs, inst=inst, H=H, y=y, out=out, ws=ws, nb=nb)
    # Training: the loss's gradient at z, and (free weights) the regularizers and fusion weights being trained.
    H, y, N0 = _uplink(case, gen)
    U, C = case["U"], case["C"]
    gz = _cn((case["n_sc"], case["n_sym"], U), gen)
    st = dict(case=case, H=H.requires_grad_(), y=y.requires_grad_(), N0=N0, gz=gz)
    if case["kind"] == "train":
        st["rho"] = (N0 / ES * (0.5 + torch.rand(C, generator=gen, device=dev))).requires_grad_()
        nu = 0.5 + torch.rand((C, U), generator=gen, device=dev)
        st["nu"] = (nu / nu.sum(0)).requires_grad_()
    return st


# ------------------------------------------------------------------------------------------- one pass

def run(st):
    case = st["case"]
    if case["kind"] == "equalize":
        o = st["out"]
        ffeq.ffeq_equalize(st["plan"], st["H"], st["y"], st["N0"], ES, o["z"], o["sigma2"], o["llr"], o.get("info"),
                           st["ws"], st["nb"])
        return o
    if case["kind"] == "uneven":
        o = st["out"]
        ffeq.ffeq_batch_equalize(st["batch"], st["H"], st["y"], o["z"], o["sigma2"], o["llr"], o["info"], st["ws"],
                                 st["nb"])
        return o
    if case["kind"] == "train":
        z = autograd.fd_equalize(st["H"], st["y"], st["rho"], st["nu"], case["C"])
        gH, gy, grho, gnu = torch.autograd.grad(z, (st["H"], st["y"], st["rho"], st["nu"]), st["gz"])
        return dict(z=z.detach(), gH=gH, gy=gy, grho=grho, gnu=gnu)
    z = autograd.fd_equalize_optimal(st["H"], st["y"], st["N0"], ES, case["C"])
    gH, gy = torch.autograd.grad(z, (st["H"], st["y"]), st["gz"])
    return dict(z=z.detach(), gH=gH, gy=gy)


# ------------------------------------------------------------------------------------------- needed work

def _system_flops(B, U, C, n_sym, arch, equalizer, iters, bits):
    """Real operations of one subcarrier: the Hermitian half of the Gram matrices, the matched filters, and per
    system one factorization, the inverse's diagonal and n_sym solves (or LAMA's products and denoisers)."""
    systems = C if arch == "fd" else 1
    f = 8 * B * (U * (U + 1) // 2 + U * n_sym)
    if equalizer in ("lmmse", "zf"):
        f += systems * (8 * U ** 3 // 3 + 8 * U * U * n_sym)
    elif equalizer == "mrc":
        f += systems * (4 * U * U + 2 * U * n_sym)
    else:
        f += systems * n_sym * (8 * U * U * iters + U * (12 * (1 << (bits // 2)) + 20) * (iters - 1))
    return f + 4 * U * n_sym * bits


def work(case):
    if case["kind"] == "uneven":
        specs = _uneven_specs(case)
        by = fl = 0
        for B, U, C, _, n_sym, _, _ in specs:
            by += 8 * (B * (U + n_sym) + U * n_sym) + 4 * U * (1 + n_sym * case["bits"]) + 4 * (C if case["arch"] == "fd" else 1)
            fl += _system_flops(B, U, C, n_sym, case["arch"], case["equalizer"], 0, case["bits"])
        return {"bytes": by, "flops": fl}
    B, U, C, n_sc, n_sym = (case[k] for k in ("B", "U", "C", "n_sc", "n_sym"))
    if case["kind"] == "equalize":
        out = 8 * U * n_sym + 4 * U * (n_sym if case["equalizer"] == "lama" else 1) + 4 * U * n_sym * case["bits"]
        out += 4 * (C if case["arch"] == "fd" else 1) if case["info"] else 0
        fl = _system_flops(B, U, C, n_sym, case["arch"], case["equalizer"], case["iters"], case["bits"])
        systems = C if case["arch"] == "fd" else 1
        # A refinement step: H [A | X], H^H of the residual, A r.
        fl += case["refine"] * (8 * B * U * (U + 2 * n_sym) + systems * 8 * U * U * n_sym)
        return {"bytes": n_sc * (8 * B * (U + n_sym) + out), "flops": n_sc * fl}
    # A training step reads H, y, dL/dz and writes z, dL/dH and dL/dy: one factorization and a solve per direction,
    # and the gradient products.
    fl = _system_flops(B, U, C, 2 * n_sym, "fd", "lmmse", 0, 0) + 8 * B * U * 4 * n_sym
    if case["kind"] == "optimal":
        fl += 8 * B * U * U * 2
    return {"bytes": n_sc * 16 * (B * (U + n_sym) + U * n_sym), "flops": n_sc * fl}


# ------------------------------------------------------------------------------------------- 64 bits

def _levels(bits):
    L = 1 << (bits // 2)
    return (torch.arange(L, device="cuda", dtype=torch.float64) * 2 - (L - 1)) * math.sqrt(ES * 1.5 / (L * L - 1))


def _llr64(z, s2, bits):
    """Max-log LLRs of Gray-labelled square QAM per axis (the other axis' distance cancels)."""
    h, lev = bits // 2, _levels(bits)
    i = torch.arange(lev.numel(), device="cuda")
    gray = i ^ (i >> 1)
    out = []
    for axis in (z.real, z.imag):
        d = (axis[..., None] - lev) ** 2
        for t in range(h):
            one = ((gray >> (h - 1 - t)) & 1).bool()
            out.append((d[..., one].amin(-1) - d[..., ~one].amin(-1)) / s2)
    return torch.stack(out, dim=-1)


def _clusters(H, y, C, arch):
    """Columns per system: Hc [n][C'][S][U], Yc [n][C'][S][n_sym] in 64 bits (C' = C for FD, 1 for PD)."""
    Cs = C if arch == "fd" else 1
    n, U, B = H.shape
    f = lambda a: a.to(torch.complex128).reshape(n, a.shape[1], Cs, B // Cs).permute(0, 2, 3, 1)  # noqa: E731
    return f(H), f(y)


def _lama64(G, b, S, N0, bits, iters):
    U = G.shape[-1]
    beta, n0, lev = U / S, N0 / S, _levels(bits)
    G, b = G / S, b / S
    s, v = torch.zeros_like(b), torch.zeros_like(b)
    phi = torch.full(b.shape[:-2] + (1, b.shape[-1]), ES, dtype=torch.float64, device=b.device)
    for t in range(iters):
        z = b + s - G @ s + v
        tau = n0 + beta * phi
        if t + 1 == iters:
            return z, tau
        mean, var = [], 0.0
        for axis in (z.real, z.imag):
            w = torch.softmax(-(axis[..., None] - lev) ** 2 / tau[..., None], dim=-1)
            m = (w * lev).sum(-1)
            mean.append(m)
            var = var + (w * (lev - m[..., None]) ** 2).sum(-1)
        new = torch.complex(mean[0], mean[1])
        phi = var.mean(dim=-2, keepdim=True)
        v = beta * phi / tau * (z - s)
        s = new


def _equalize64(H, y, N0, C, arch, equalizer, bits, iters):
    Hc, Yc = _clusters(H, y, C, arch)
    G, b = Hc.mH @ Hc, Hc.mH @ Yc
    U = G.shape[-1]
    if equalizer == "lama":
        z, s2 = _lama64(G, b, Hc.shape[2], N0, bits, iters)
        s2 = s2.expand(z.shape)
    elif equalizer == "mrc":
        g = torch.diagonal(G, dim1=-2, dim2=-1).real
        other = (G.abs() ** 2).sum(-1) - g ** 2
        z, s2 = b / g[..., None], ((N0 * g + ES * other) / g ** 2)[..., None]
    else:
        rho = N0 / ES if equalizer == "lmmse" else 0.0
        A = torch.linalg.inv(G + rho * torch.eye(U, dtype=G.dtype, device=G.device))
        a = torch.diagonal(A, dim1=-2, dim2=-1).real
        mu = 1.0 - rho * a
        z, s2 = (A @ b) / mu[..., None], (N0 * a / mu)[..., None]
    w = 1.0 / s2
    zf, s2f = (w * z).sum(1) / w.sum(1), 1.0 / w.sum(1)                 # [n][U][n_sym], [n][U][1 or n_sym]
    zf, s2f = zf.mT, s2f.mT
    return dict(z=zf, sigma2=s2f if equalizer == "lama" else s2f[:, 0], llr=_llr64(zf, s2f, bits))


def _train64(st):
    """The adjoint in closed form is what is measured; here autograd differentiates 64-bit torch."""
    case = st["case"]
    H = st["H"].detach().to(torch.complex128).requires_grad_()
    y = st["y"].detach().to(torch.complex128).requires_grad_()
    Hc, Yc = _clusters(H, y, case["C"], "fd")
    eye = torch.eye(case["U"], dtype=torch.complex128, device="cuda")
    G, b = Hc.mH @ Hc, Hc.mH @ Yc
    if case["kind"] == "train":
        rho, nu = (st[k].detach().double().requires_grad_() for k in ("rho", "nu"))
        X = torch.linalg.solve(G + rho[:, None, None] * eye, b)
        z = (nu[..., None] * X).sum(1).mT
        g = torch.autograd.grad(z, (H, y, rho, nu), st["gz"].to(torch.complex128))
        return dict(z=z.detach(), gH=g[0], gy=g[1], grho=g[2], gnu=g[3])
    rho = st["N0"] / ES
    A = torch.linalg.inv(G + rho * eye)
    w = 1.0 / torch.diagonal(A, dim1=-2, dim2=-1).real
    z = ((w[..., None] * (A @ b)).sum(1) / (w - rho).sum(1)[..., None]).mT
    g = torch.autograd.grad(z, (H, y), st["gz"].to(torch.complex128))
    return dict(z=z.detach(), gH=g[0], gy=g[1])


def exact(case, seed):
    st = prepare(case, seed)
    if case["kind"] in ("train", "optimal"):
        return _train64(st)
    if case["kind"] == "equalize":
        n, parts = 300, []
        for k in range(0, case["n_sc"], n):
            parts.append(_equalize64(st["H"][k:k + n], st["y"][k:k + n], st["N0"], case["C"], case["arch"],
                                     case["equalizer"], case["bits"], case["iters"]))
        out = {k: torch.cat([p[k] for p in parts]) for k in parts[0]}
    else:
        out = {k: torch.zeros(v.shape, dtype=torch.complex128 if v.is_complex() else torch.float64, device="cuda")
               for k, v in st["out"].items() if k != "info"}
        offs = {"z": "z_off", "sigma2": "sigma2_off", "llr": "llr_off"}
        for (B, U, C, _, n_sym, N0, _), it in zip(st["specs"], st["inst"]):
            H = st["H"][it.h_off:it.h_off + U * B].view(1, U, B)
            y = st["y"][it.y_off:it.y_off + n_sym * B].view(1, n_sym, B)
            got = _equalize64(H, y, N0, C, case["arch"], case["equalizer"], case["bits"], 0)
            for k, v in got.items():
                at = getattr(it, offs[k])
                out[k][at:at + v.numel()] = v.reshape(-1)
    if "info" in st["out"]:
        out["info"] = None
    return out
