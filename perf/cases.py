"""The calls a user of this library makes, as timed cases.

Each case is one call (or one call with its gradient) through
paper_1208_3210_gb300.lindhard: a plan made once for its grid, then Im chi (or
Im chi_T, S(q, w), the adjoint, the Kramers-Kronig pass) for the inputs at
hand.  Sizes are the workloads of paper_1208_3210_gb300/workloads.py, of the
tests and of bench.py, and generic ones between them.
"""
import math

import torch

from paper_1208_3210_gb300 import lindhard as lh
from paper_1208_3210_gb300 import workloads as wl


def _case(call, zones, npz, n_eps, e_max, name=None, **over):
    c = dict(call=call, zones=zones, npz=npz, n_eps=n_eps, e_max=e_max, n_omega=n_eps // 2, q_extent=zones * npz,
             quantity=lh.IMCHI, gamma=0.05, ff_a=1.0, kT=0.0, plan="default")
    c.update(over)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the reduced-zone check every user starts with: launches and the mu solve
        _case("imchi", 1, 32, 48, 1.0, "one_zone", ff_a=0.0),
        # every lag of an odd-sized grid (what the sum rule needs), plan without tuning
        _case("imchi", 3, 50, 201, 2.0, "all_lags", q_extent=300, ff_a=0.5),
        # the extended-zone workload, tuned plan
        _case("imchi", 4, 64, 256, 2.0, "extended", plan="autotune"),
        # the large extended-zone workload, tuned plan (the benchmark's headline)
        _case("imchi", 8, 128, 512, 3.0, "large", gamma=0.03, plan="autotune"),
        # a spectral function from elsewhere (no symmetry) on the extended grid
        _case("given", 4, 64, 256, 2.0, "given_spectrum", plan="autotune"),
        # finite temperature on the extended grid
        _case("imchi", 4, 64, 256, 2.0, "thermal", quantity=lh.IMCHI_T, kT=0.025, plan="autotune"),
        # the structure factor on a ragged grid, plan without tuning
        _case("imchi", 5, 36, 150, 2.0, "structure_factor", quantity=lh.SQW, kT=0.05),
        # one step of a fit of the band to a weighted loss: value and gradient by autograd
        _case("fit", 4, 64, 256, 2.0, "fit_step", plan="autotune"),
        # dL/dA over the whole large grid (for a chain rule of the caller's own)
        _case("adjoint", 8, 128, 512, 3.0, "adjoint_large", gamma=0.03, plan="autotune"),
        # Re chi and chi_RPA of the large output
        _case("kk_rpa", 8, 128, 512, 3.0, "kk_rpa_large"),
        # many small and middle instances of mixed size in one call (a captured graph)
        dict(name="batch_64", call="batch", count=64, mix=0, plan="graph"),
        # double precision, as used to tell rounding from method errors
        _case("double", 2, 32, 128, 2.0, "double", ff_a=0.8, gamma=0.08),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["imchi", "imchi", "imchi", "thermal", "thermal", "given", "fit", "adjoint", "kk_rpa", "batch",
                       "double"])
    if call == "batch":
        return dict(call="batch", count=rng.randint(3, 24), mix=rng.randint(1, 1 << 20),
                    plan=rng.choice(["default", "autotune", "concurrent", "graph", "persistent"]))
    ff_a = rng.choice([0.0, round(rng.uniform(0.3, 1.2), 3), 1.0])
    gamma = round(rng.uniform(0.02, 0.2), 4)
    plan = rng.choice(["default", "autotune"])
    e_max = round(rng.uniform(1.5, 3.0), 2)
    if call == "double":
        zones = rng.randint(2, 4)
        return _case("double", zones, 2 * rng.randint(4, 128 // (2 * zones)), rng.randint(16, 200), e_max,
                     gamma=gamma, ff_a=ff_a)
    if call == "imchi" and rng.random() < 0.25:   # the reduced zone
        n_eps = _log_int(rng, 24, 512)
        return _case("imchi", 1, rng.choice([16, 32, 64, 128, 256]), n_eps, e_max, gamma=gamma, ff_a=0.0, plan=plan)
    zones = rng.randint(2, 8)
    npz = 2 * max(2, _log_int(rng, 48, 640) // (2 * zones))
    N = zones * npz
    n_eps = _log_int(rng, 24, 512)
    extent = rng.choice([N, N, N, 2 * N, 2 * rng.randint(1, N // 2)])
    if call == "thermal":
        return _case("imchi", zones, npz, n_eps, e_max, q_extent=extent, gamma=gamma, ff_a=ff_a, plan=plan,
                     quantity=rng.choice([lh.IMCHI_T, lh.SQW]), kT=round(rng.uniform(0.01, 0.2), 4))
    if call in ("fit", "adjoint"):
        return _case(call, zones, npz, n_eps, e_max, gamma=gamma, ff_a=ff_a, plan=plan)
    if call == "kk_rpa":
        return _case(call, zones, npz, n_eps, e_max, gamma=gamma, ff_a=ff_a)
    n_omega = rng.choice([n_eps // 2, n_eps // 2, rng.randint(1, n_eps)])
    return _case(call, zones, npz, n_eps, e_max, q_extent=extent, n_omega=n_omega, gamma=gamma, ff_a=ff_a, plan=plan)


# --- inputs -----------------------------------------------------------------------


def _grids(case):
    if case["call"] == "batch":
        return wl.batched_workload(case["count"], case["mix"])[0]
    return [wl.grid_params(case["zones"], case["npz"], case["n_eps"], case["e_max"], case["n_omega"],
                           case["q_extent"], quantity=case["quantity"])]


def _bands(case, seed):
    """Bands of this seed: doping, broadening and hoppings around the case's."""
    g = torch.Generator().manual_seed(seed)
    if case["call"] == "batch":
        nominal = wl.batched_workload(case["count"], case["mix"])[1]
    else:
        nominal = [wl.band_params(filling=1.12, gamma=case["gamma"], ff_a=case["ff_a"], kT=case["kT"])]
    out = []
    for b in nominal:
        r = (2 * torch.rand(5, generator=g, dtype=torch.float64) - 1).tolist()
        out.append(dict(b, filling=b["filling"] + 0.04 * r[0], gamma=b["gamma"] * (1 + 0.1 * r[1]),
                        t=b["t"] * (1 + 0.03 * r[2]), tp=b["tp"] * (1 + 0.03 * r[3]), tpp=b["tpp"] * (1 + 0.03 * r[4])))
    return out


def _weights(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand(case["q_extent"] ** 2 * case["n_omega"], generator=g, device="cuda")


def _given(case, seed):
    """A spectral function with no lattice symmetry: a band's, times a noisy profile."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    A = _spectral(case, _bands(case, seed)[0]).float()
    return (A * (0.5 + torch.rand(A.shape, generator=g, device="cuda"))).contiguous()


def _response(case, seed):
    """An Im chi block as a forward call leaves it: negative, zero at w = 0, a
    peak that disperses and decays with q."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    Q, n = case["q_extent"], case["n_omega"]
    s = (torch.arange(Q, device="cuda") - Q // 2) * (2 * math.pi / case["npz"])
    q = torch.sqrt(s[:, None] ** 2 + s[None, :] ** 2)
    w = torch.arange(n, device="cuda") / n
    centre = (0.2 + 0.5 * torch.sin(0.5 * q) ** 2)[..., None]
    im = -torch.exp(-q * q / 16)[..., None] * w / ((w - centre) ** 2 + 0.01)
    return (im * (0.9 + 0.2 * torch.rand(im.shape, generator=g, device="cuda"))).contiguous()


def prepare(case, seed):
    call = case["call"]
    state = dict(call=call)
    plan = lh.Plan(_grids(case), precision=lh.FP64 if call == "double" else lh.FP32,
                   backward=call in ("fit", "adjoint"), autotune=case["plan"] in ("autotune", "graph"),
                   concurrent=case["plan"] == "concurrent", graph=case["plan"] == "graph",
                   persistent=case["plan"] == "persistent")
    state["plan"] = plan
    if call == "kk_rpa":
        state["imchi"] = _response(case, seed)
        return state
    if call == "given":
        state["A"] = _given(case, seed)
    bands = _bands(case, seed)
    if call in ("fit", "adjoint"):   # a gradient is taken at a given mu
        mu = _mu(case["npz"], bands[0])
        bands = [dict(bands[0], mu=mu, filling=float("nan"))]
        state["w"] = _weights(case, seed)
    state["bands"] = bands
    if call == "fit":
        b = bands[0]
        state["params"] = torch.tensor([[b[k] for k in lh.PARAM_NAMES]], requires_grad=True)
    elif call == "adjoint":
        state["dA"] = torch.empty(plan.a_elems(), device="cuda")
    else:
        state["out"] = torch.empty(plan.out_elems(), dtype=torch.float64 if call == "double" else torch.float32,
                                   device="cuda")
        state["mu"] = torch.empty(plan.batch, dtype=torch.float64, device="cuda")
    return state


def run(state):
    plan, call = state["plan"], state["call"]
    if call == "kk_rpa":
        return plan.kk_rpa(state["imchi"], v0=0.05)
    if call == "given":
        return plan.imchi(out=state["out"], A_in=state["A"])
    if call == "fit":
        chi = lh.ImChiFunction.apply(state["params"], plan, state["bands"])
        loss = (state["w"] * chi).sum()
        grad, = torch.autograd.grad(loss, state["params"])
        return chi.detach(), grad
    if call == "adjoint":
        return plan.backward(state["w"], bands=state["bands"], dA=state["dA"])[0]
    plan.imchi(state["bands"], out=state["out"], mu_out=state["mu"])
    return state["out"], state["mu"]


# --- the work of a call -----------------------------------------------------------


def work(case):
    """Bytes in and out once, and the operations of the correlation by FFT
    (2.5 n log2 n per real transform of n points of the zero-padded volume,
    three of them forward, five more with the adjoint).  A band's spectral
    function is even in p_x and p_y and symmetric under their exchange, so one
    eighth of its volume is independent."""
    total_b = total_f = 0.0
    for g in _grids(case):
        N, Q, ne, nw = g["zones"] * g["npz"], g["q_extent"], g["n_eps"], g["n_omega"]
        P = N if g["zones"] == 1 else N + Q // 2
        E = ne if g.get("quantity", 0) == lh.IMCHI else ne + nw
        fft = 2.5 * P * P * E * math.log2(P * P * E)
        out, a = 4.0 * Q * Q * nw, 4.0 * N * N * ne
        call = case["call"]
        if call == "kk_rpa":
            total_b += 4 * out                       # Im chi in, Re chi and complex chi_RPA out
            total_f += Q * Q * nw * (nw / 2.0 * 2 + 20)
        elif call == "given":
            total_b += a + out
            total_f += 3 * fft
        elif call == "fit":
            total_b += 2 * out                       # the weights in, Im chi out
            total_f += 6 * fft / 8
        elif call == "adjoint":
            total_b += out + a                       # the weights in, dL/dA out
            total_f += 3 * fft + 2 * fft / 8         # the weights have no symmetry
        else:
            total_b += 2 * out if call == "double" else out
            total_f += 3 * fft / 8
    return dict(bytes=total_b, flops=total_f)


# --- the same in 64 bits, without the library ------------------------------------------


def _axis(npz, N):
    return (torch.arange(N, dtype=torch.float64, device="cuda") - N // 2) * (2 * math.pi / npz)


def _band_energy(b, p):
    """Band energy on the grid p x p, mu not subtracted, and its derivatives by t, t', t''."""
    c1, c2 = torch.cos(p), torch.cos(2 * p)
    dt = -2 * (c1[:, None] + c1[None, :])
    dtp = -4 * c1[:, None] * c1[None, :]
    dtpp = -2 * (c2[:, None] + c2[None, :])
    return b["t"] * dt + b["tp"] * dtp + b["tpp"] * dtpp, (dt, dtp, dtpp)


def _mu(npz, b):
    """Chemical potential of the band's filling, by bisection."""
    e0 = _band_energy(b, _axis(npz, npz))[0]
    lo, hi = -1e3, 1e3
    for _ in range(80):
        mid = 0.5 * (lo + hi)
        n = 2.0 * (0.5 - torch.atan((e0 - mid) / b["gamma"]) / math.pi).mean().item()
        lo, hi = (mid, hi) if n < b["filling"] else (lo, mid)
    return 0.5 * (lo + hi)


def _energies(g):
    de = 2 * g["e_max"] / g["n_eps"]
    return -g["e_max"] + (torch.arange(g["n_eps"], dtype=torch.float64, device="cuda") + 0.5) * de


def _amplitude(g, b):
    p = _axis(g["npz"], g["zones"] * g["npz"])
    m = torch.exp(-p * p * b["ff_a"] ** 2 / 8)
    return (m[:, None] * m[None, :])[..., None]


def _spectral(g, b):
    mu = b["mu"] if math.isnan(b["filling"]) else _mu(g["npz"], b)
    xi = _band_energy(b, _axis(g["npz"], g["zones"] * g["npz"]))[0] - mu
    x = (_energies(g) - xi[..., None]).square_().add_(b["gamma"] ** 2).reciprocal_()
    return x.mul_(_amplitude(g, b) * (b["gamma"] / math.pi))


def _split(g, A, kT):
    """Occupied and empty parts of A."""
    if g.get("quantity", lh.IMCHI) == lh.IMCHI:
        occ = (torch.arange(g["n_eps"], device="cuda") < g["n_eps"] // 2).double()
    else:
        occ = torch.sigmoid(-_energies(g) / kT)
    return A * occ, A * (1 - occ)


def _lengths(g):
    N, Q = g["zones"] * g["npz"], g["q_extent"]
    P = N if g["zones"] == 1 else N + Q // 2
    if P > 64:
        P = -(-P // 16) * 16 if g["zones"] > 1 else P
    E = g["n_eps"] + (0 if g.get("quantity", lh.IMCHI) == lh.IMCHI else g["n_eps"])
    return P, E + E % 2


def _prefactor(g):
    c = 2 * g["e_max"] / g["n_eps"] / (2 * math.pi) / g["npz"] ** 2
    return c / math.pi if g.get("quantity", lh.IMCHI) == lh.SQW else -c


def _spectra(x, E):
    """Half spectra along the energy axis, frequencies first."""
    return torch.fft.rfft(x, n=E, dim=2).permute(2, 0, 1)


def _lags(g, P):
    return (torch.arange(g["q_extent"], device="cuda") - g["q_extent"] // 2) % P


def _correlate(g, A, kT):
    """The grid's quantity for the spectral function A, [Q][Q][n_omega]."""
    P, E = _lengths(g)
    a, b = (_spectra(x, E) for x in _split(g, A, kT))
    l = _lags(g, P)
    out = torch.empty((E // 2 + 1, len(l), len(l)), dtype=torch.complex128, device="cuda")
    for k in range(0, E // 2 + 1, 16):
        prod = torch.fft.fft2(a[k:k + 16], s=(P, P)).conj_physical_() * torch.fft.fft2(b[k:k + 16], s=(P, P))
        if g.get("quantity", lh.IMCHI) == lh.IMCHI_T:
            prod = prod - prod.conj()
        out[k:k + 16] = torch.fft.ifft2(prod)[:, l][:, :, l]
    del a, b
    r = torch.fft.irfft(out.permute(1, 2, 0), n=E, dim=2)[..., :g["n_omega"]]
    return r.mul_(_prefactor(g)).contiguous()


def _grad_A(g, A, w):
    """dL/dA of L = sum w Im chi (T = 0)."""
    N = g["zones"] * g["npz"]
    P, E = _lengths(g)
    a, b = (_spectra(x, E) for x in _split(g, A, 0.0))
    W = _spectra(w.double(), E)
    l = _lags(g, P)
    h = torch.empty_like(a)
    for k in range(0, E // 2 + 1, 16):
        full = torch.zeros((W[k:k + 16].shape[0], P, P), dtype=torch.complex128, device="cuda")
        full[:, l[:, None], l[None, :]] = W[k:k + 16]
        f = torch.fft.fft2(full)
        occ = torch.fft.ifft2(f.conj() * torch.fft.fft2(b[k:k + 16], s=(P, P)))[:, :N, :N]
        h[k:k + 16] = torch.fft.ifft2(f * torch.fft.fft2(a[k:k + 16], s=(P, P)))[:, :N, :N]
        b[k:k + 16] = occ
    del a, W
    J0, n = g["n_eps"] // 2, g["n_eps"]
    out = torch.empty((N, N, n), dtype=torch.float64, device="cuda")
    for i in range(0, N, 128):
        out[i:i + 128, :, :J0] = torch.fft.irfft(b[:, i:i + 128].permute(1, 2, 0), n=E, dim=2)[..., :J0]
        out[i:i + 128, :, J0:] = torch.fft.irfft(h[:, i:i + 128].permute(1, 2, 0), n=E, dim=2)[..., J0:n]
    return out.mul_(_prefactor(g))


def _grad_params(g, b, G):
    """Chain rule from dL/dA to (t, t', t'', mu, gamma)."""
    e0, d = _band_energy(b, _axis(g["npz"], g["zones"] * g["npz"]))
    amp, gam, out = _amplitude(g, b) / math.pi, b["gamma"], torch.zeros(5, dtype=torch.float64, device="cuda")
    for i in range(0, e0.shape[0], 128):
        x = _energies(g) - (e0[i:i + 128] - b["mu"])[..., None]
        D = (x * x + gam * gam).square_()
        Gi = G[i:i + 128] * amp[i:i + 128] / D
        s = (Gi * (2 * gam) * x).sum(2)
        out += torch.stack([(s * d[0][i:i + 128]).sum(), (s * d[1][i:i + 128]).sum(), (s * d[2][i:i + 128]).sum(),
                            -s.sum(), (Gi * (x * x - gam * gam)).sum()])
    return out


def exact(case, seed):
    call, grids = case["call"], _grids(case)
    g = grids[0]
    if call == "kk_rpa":
        im = _response(case, seed).double()
        n, Q = g["n_omega"], g["q_extent"]
        m, k = torch.arange(n, device="cuda")[:, None], torch.arange(n, device="cuda")[None, :]
        odd = ((k - m) % 2 != 0) & (k >= 1)
        W = torch.where(odd, 4 / math.pi * k.double() / torch.where(odd, k * k - m * m, 1).double(), 0.0)
        re = (im.reshape(-1, n) @ W.T).reshape(im.shape)
        s = (torch.arange(Q, dtype=torch.float64, device="cuda") - Q // 2) * (2 * math.pi / g["npz"])
        chi = torch.complex(re, im)
        q2 = s[:, None] ** 2 + s[None, :] ** 2
        V = 0.05 / torch.where(q2 > 0, q2, 1.0)
        rpa = chi / (1 - V[..., None] * chi)
        rpa[q2 == 0] = 0
        return re, rpa
    if call == "given":
        return _correlate(g, _given(case, seed).double(), 0.0).reshape(-1)
    bands = _bands(case, seed)
    mus = [_mu(x["npz"], b) for x, b in zip(grids, bands)]
    if call in ("fit", "adjoint"):
        b = dict(bands[0], mu=mus[0], filling=float("nan"))
        if call == "fit":   # the parameters as the tensor holds them
            b.update({k: float(torch.tensor(b[k])) for k in lh.PARAM_NAMES})
        A = _spectral(g, b)
        chi = _correlate(g, A, 0.0).reshape(-1) if call == "fit" else None
        G = _grad_A(g, A, _weights(case, seed).reshape(g["q_extent"], g["q_extent"], g["n_omega"]))
        del A
        return (chi, _grad_params(g, b, G).reshape(1, 5)) if call == "fit" else G.reshape(-1)
    out = [_correlate(x, _spectral(x, dict(b, mu=mu, filling=float("nan"))), b.get("kT", 0.0)).reshape(-1)
           for x, b, mu in zip(grids, bands, mus)]
    return torch.cat(out), torch.tensor(mus, dtype=torch.float64, device="cuda")
