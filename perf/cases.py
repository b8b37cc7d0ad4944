"""The work that a program has this library do, as cases that can be timed.

A case is one pass of such a program through the public entry points: a sweep of a batch
of chains with its log-weights (and, where a program reads them every time, observables or
the configuration), a local-update sweep, or one differentiation of log Z.  Sizes are
those of the benchmark family and of the paper's runs; `draw` spreads over the same
ranges: every supported lattice size, odd slice counts and worldline counts, blocks,
permutations, attractive U, both precisions.

A case's `Nsig` is the number of worldlines per spin (filling = 2 Nsig / N) and `M` the
number of slices (beta = M dtau); t = 1.
"""
import math

import numpy as np
import torch

from paper_2510_13866_gb300 import Lattice, log_weight

# batch of chains of uneven size: the benchmark's ranges of L, beta, U and filling
MIX_L = (8, 12, 16, 24, 32, 48)
MIX_BETA = (2.0, 4.0, 6.0)
MIX_U = (2.0, 4.0, 8.0)
MIX_FILL = (0.5, 0.875, 1.0)
SIZES = (2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64, 128)

DEFAULTS = dict(kind="sweep", L=8, chains=1, M=20, Nsig=1, U=4.0, dtau=0.05, precision="fp32", block=0, perm=False,
                open=False, stencil=False, observables=False, configuration=False)


def _case(name=None, **kw):
    c = dict(DEFAULTS)
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # a first look at the model: one 4 x 4 chain, every configuration read back
        _case("sweep_L4", L=4, M=20, Nsig=8, dtau=0.1, configuration=True),
        # the paper's runs (beta = 32, blocks of 32 slices): one chain, observables each sweep
        _case("sweep_paper_L8", L=8, M=1024, Nsig=32, U=20.0, dtau=1 / 32, block=32, observables=True),
        # a fermionic run below half filling: permutations and the momentum distribution
        _case("sweep_perm_nk_L12", L=12, chains=32, M=120, Nsig=63, perm=True, open=True, observables=True),
        # attractive U: the continuous field
        _case("sweep_attractive_L16", L=16, chains=32, M=80, Nsig=112, U=-4.0),
        # the double-precision form, the check on a single-precision run
        _case("sweep_fp64_L16", L=16, chains=4, M=80, Nsig=128, precision="fp64", configuration=True),
        # production at 32 x 32: the benchmark's batch of 64 chains
        _case("sweep_L32", L=32, chains=64, M=80, Nsig=512),
        # a parameter scan: 256 chains of uneven size, temperature and filling in one launch
        _case("sweep_mixed", kind="mixed", L=0, chains=256, M=0, Nsig=0),
        # large lattices
        _case("sweep_L64", L=64, chains=16, M=160, Nsig=2048),
        _case("sweep_L128", L=128, chains=2, M=160, Nsig=4096),
        # local link updates between FFBS sweeps, observables each time
        _case("local_L32", kind="local", L=32, chains=64, M=80, Nsig=512, observables=True),
        # a training step on log Z: gradients to the log-potential and the hopping
        _case("adjoint_L16", kind="adjoint", L=16, chains=128, M=80, Nsig=128),
        _case("adjoint_L64", kind="adjoint", L=64, chains=2, M=40, Nsig=512),
    ]


# worldline-slice-sites of the largest listed pass (sweep_L64); a drawn case stays below
_TOP = 16 * 2 * 2048 * 160 * 4096


def draw(rng):
    kind = rng.choice(("sweep", "sweep", "sweep", "sweep", "sweep", "local", "adjoint", "adjoint", "mixed"))
    if kind == "mixed":
        return _case(kind="mixed", L=0, chains=int(round(math.exp(rng.uniform(math.log(6), math.log(256))))), M=0, Nsig=0)
    L = rng.choice(SIZES)
    N = L * L
    precision = "fp64" if kind == "sweep" and L <= 24 and rng.random() < 0.15 else "fp32"
    M = int(round(math.exp(rng.uniform(math.log(4), math.log(200 if L > 4 else 80)))))
    if L > 32:
        M = min(M, 160)
    Nsig = max(1, min(N, int(round(N / 2 * rng.choice((1.0, 1.0, 0.875, 0.5, rng.uniform(0.02, 1.0)))))))
    unit = 2 * Nsig * M * N * (30 if precision == "fp64" else 8 if kind == "adjoint" else 1)
    most = max(1, min(512, int(_TOP / 4 / unit)))
    chains = max(1, int(round(math.exp(rng.uniform(0.0, math.log(most))))))
    U = rng.choice((2.0, 4.0, 4.0, 8.0, 20.0, -4.0))
    dtau = rng.choice((0.05, 0.05, 0.1, 1 / 32))
    block = 0
    perm = open_ = stencil = False
    if kind == "sweep":
        if M >= 40 and rng.random() < 0.25:
            block = rng.choice((16, 32, 37))
        perm = rng.random() < 0.15
        open_ = rng.random() < 0.15
        stencil = L <= 32 and rng.random() < 0.1
    obs = kind == "local" or open_ or rng.random() < 0.3
    conf = kind == "sweep" and U > 0 and chains * Nsig * M <= 200_000 and rng.random() < 0.6
    return _case(kind=kind, L=L, chains=chains, M=M, Nsig=Nsig, U=U, dtau=dtau, precision=precision, block=block,
                 perm=perm, open=open_, stencil=stencil, observables=obs and kind != "adjoint", configuration=conf)


# --- inputs ---------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _chains(case, seed):
    """(L, M, Nsig, U, dtau, chain seed) of every chain."""
    first = 1000 * (int(seed) % 1_000_000)
    if case["kind"] != "mixed":
        return [(case["L"], case["M"], case["Nsig"], case["U"], case["dtau"], first + c) for c in range(case["chains"])]
    # sizes and parameters are the case's own (the same for every seed)
    r = np.random.RandomState(1)
    out = []
    for c in range(case["chains"]):
        L, beta, U, fill = (v[r.randint(len(v))] for v in (MIX_L, MIX_BETA, MIX_U, MIX_FILL))
        out.append((L, int(round(beta / 0.05)), int(round(fill * L * L / 2)), U, 0.05, first + c))
    return out


def _worldlines(gen, L, M, Nsig, dtau):
    """Closed worldlines [2, Nsig, M]: discrete bridges of the hopping's step rate from distinct
    sites (the down spin on the sites that the up spin leaves free)."""
    N = L * L
    sites = torch.randperm(N, generator=gen, device="cuda")
    start = torch.stack([sites[:Nsig], sites.flip(0)[:Nsig]])
    pos = []
    for first in (start % L, start // L):
        u = torch.rand((2, Nsig, M), generator=gen, device="cuda", dtype=torch.float64)
        step = (u < dtau).double() - (u > 1 - dtau).double()
        w = torch.cumsum(step, 2)
        ramp = torch.arange(1, M + 1, device="cuda", dtype=torch.float64) / M
        pos.append((first[..., None] + torch.round(w - w[..., -1:] * ramp).long()) % L)
    return pos[0] + L * pos[1]


def _counts(x, M, N):
    """Occupation [M, N] of one spin's worldlines [Nsig, M]."""
    idx = (torch.arange(M, device=x.device)[None, :] * N + x).reshape(-1)
    return torch.bincount(idx, minlength=M * N).reshape(M, N).double()


def _hirsch_lambda(U, dtau):
    return math.acosh(math.exp(0.5 * dtau * U))


def _configuration(case, seed):
    """Per chain: worldlines and a field drawn from its conditional given them."""
    gen = _generator(seed)
    for L, M, Nsig, U, dtau, cs in _chains(case, seed):
        N = L * L
        x = _worldlines(gen, L, M, Nsig, dtau)
        up, dn = _counts(x[0], M, N), _counts(x[1], M, N)
        if U < 0:
            a = math.sqrt(-U * dtau)
            field = a * (up + dn - 0.5) + torch.randn((M, N), generator=gen, device="cuda", dtype=torch.float64)
        else:
            p = torch.sigmoid(2 * _hirsch_lambda(U, dtau) * (up - dn))
            field = 2.0 * (torch.rand((M, N), generator=gen, device="cuda", dtype=torch.float64) < p).double() - 1.0
        yield (L, M, Nsig, U, dtau, cs), x, field


def _log_potential(field, U, dtau):
    """log W of both spins [2, M, N]."""
    if U < 0:
        v = math.sqrt(-U * dtau) * field
        return torch.stack([v, v])
    v = _hirsch_lambda(U, dtau) * field
    return torch.stack([v, -v])


def _trained(case, seed):
    """The log-potential of a training step: log W of the fields, moved by earlier steps."""
    gen = _generator(int(seed) + 77)
    out = []
    for (L, M, Nsig, U, dtau, cs), x, field in _configuration(case, seed):
        v = _log_potential(field, U, dtau)
        out.append((v + 0.1 * torch.randn(v.shape, generator=gen, device="cuda", dtype=torch.float64)).float())
    return out


def prepare(case, seed):
    chains = _chains(case, seed)
    lat = Lattice([c[0] for c in chains], [c[5] for c in chains], precision=case["precision"])
    for i, (L, M, Nsig, U, dtau, cs) in enumerate(chains):
        lat.set_params(1.0, U, M * dtau, dtau, 2 * Nsig / (L * L), chain=i)
    if case["block"]:
        lat.set_block(case["block"])
    if case["perm"]:
        lat.set_permutations(True)
    if case["open"]:
        lat.set_measure_open(True)
    if case["stencil"]:
        lat.set_conv("stencil")
    for i, (c, x, field) in enumerate(_configuration(case, seed)):
        if c[3] < 0:
            lat.set_sigma(i, field.cpu().numpy())
            lat.set_state(i, x=x.int().cpu().numpy())
        else:
            lat.set_state(i, s=field.to(torch.int8).cpu().numpy(), x=x.int().cpu().numpy())
    state = dict(case=case, lat=lat)
    if case["kind"] == "adjoint":
        state["v"] = torch.cat([v.reshape(-1) for v in _trained(case, seed)]).requires_grad_(True)
        state["t"] = torch.tensor(1.0, requires_grad=True)
    return state


# --- one pass -------------------------------------------------------------------------
def run(state):
    case, lat = state["case"], state["lat"]
    if case["kind"] == "adjoint":
        v, t = state["v"], state["t"]
        v.grad = t.grad = None
        logz = log_weight(lat, v, t)
        logz.sum().backward()
        return dict(logz=logz.detach(), dv=v.grad, dt=t.grad)
    out = {}
    if case["kind"] == "local":
        lat.local_sweep(1)
    else:
        out["logw"] = np.concatenate([w.reshape(-1) for w in lat.sweep(1, logw=True)])
    if case["observables"]:
        obs = lat.measure()
        for key in obs[0]:
            out[key] = np.concatenate([np.atleast_1d(np.asarray(o[key])) for o in obs])
    if case["open"]:
        pairs = lat.measure_open()
        out["nk"] = np.concatenate([p[0] for p in pairs])
        out["one_body"] = np.concatenate([p[1] for p in pairs])
    if case["configuration"]:
        states = [lat.get_state(c) for c in range(case["chains"])]
        out["s"] = np.concatenate([s[0].reshape(-1) for s in states])
        out["x"] = np.concatenate([s[1].reshape(-1) for s in states])
        out["anchor"] = np.array([s[2] for s in states])
    return out


# --- the work a pass cannot do without ---------------------------------------------------
def work(case):
    flops = nbytes = 0.0
    esz = 8 if case["precision"] == "fp64" else 4
    for L, M, Nsig, U, dtau, _ in _chains(case, 0):
        N = L * L
        ps = 2.0 * Nsig * M  # worldline-slices
        filt = ps * (5 * N * math.log2(N) + 4 * N)
        field = M * N * (8.0 if U < 0 else 0.125)
        paths = 2.0 * ps
        if case["kind"] == "adjoint":
            # log Z and its adjoint: the filter, its recomputation and a reverse filter
            flops += 3 * filt
            nbytes += 2 * (2.0 * M * N * esz) + paths + 24
        elif case["kind"] == "local":
            flops += ps * 20 + 2.0 * M * N
            nbytes += 2 * (field + paths) + (16.0 * N if case["observables"] else 0)
        else:
            flops += filt + ps * 4 * N  # the filter, and a CDF per drawn slice
            nbytes += 2 * (field + paths) + 16.0 * Nsig + (16.0 * N if case["observables"] else 0)
    return {"bytes": nbytes, "flops": flops}


# --- the same numbers in 64 bits -----------------------------------------------------------
def _ring(L, dtau):
    """exp(dtau A) of the ring (t = 1) in 64 bits, and its derivative by t."""
    a = np.zeros((L, L))
    for i in range(L):
        a[i, (i + 1) % L] += 1.0
        a[i, (i - 1) % L] += 1.0
    w, q = np.linalg.eigh(a)
    g = (q * np.exp(dtau * w)) @ q.T
    dg = (q * (dtau * w * np.exp(dtau * w))) @ q.T
    return torch.from_numpy(g).cuda(), torch.from_numpy(dg).cuda()


def _propagate(f, g):
    """G * f for messages [..., L, L]: two dense ring products, or for wide lattices the same
    product in momentum space."""
    L = f.shape[-1]
    if L < 64:
        return g @ f @ g
    gh = torch.fft.rfft2(g[0][:, None] * g[0][None, :])
    return torch.fft.irfft2(torch.fft.rfft2(f) * gh, s=(L, L))


def _anchor(seed, M):
    word = np.random.Philox(counter=((2 << 128) - 1), key=int(seed)).random_raw(1)[0]
    return min(M - 1, int((int(word) >> 11) * 2.0**-53 * M))


def _filter_logw(case, seed):
    """Log-weights of the first sweep: per chain [2, Nsig]."""
    out = []
    for (L, M, Nsig, U, dtau, cs), x, field in _configuration(case, seed):
        N = L * L
        g, _ = _ring(L, dtau)
        w = torch.exp(_log_potential(field, U, dtau))  # [2, M, N]
        a = _anchor(cs, M)
        B = case["block"] if 0 < case["block"] < M else M
        logw = torch.zeros((2, Nsig), dtype=torch.float64, device="cuda")
        lengths = {}
        for b in range((M + B - 1) // B):  # blocks of one length go together
            lengths.setdefault(min(B, M - b * B), []).append((a + b * B) % M)
        most = max(1, int(2e8 / N))  # messages held at once
        for length, starts in lengths.items():
            st = torch.tensor(starts, device="cuda")
            for sg in range(2):
                x0 = x[sg][:, st].reshape(-1)                       # held first and last sites
                x1 = x[sg][:, (st + length) % M].reshape(-1)
                at = st.repeat(Nsig)
                for k in range(0, x0.numel(), most):
                    i0, i1, s0 = x0[k:k + most], x1[k:k + most], at[k:k + most]
                    f = torch.zeros((i0.numel(), N), dtype=torch.float64, device="cuda")
                    f.scatter_(1, i0[:, None], w[sg][s0 % M].gather(1, i0[:, None]))
                    norm = torch.zeros(i0.numel(), dtype=torch.float64, device="cuda")
                    for i in range(length):
                        f = _propagate(f.view(-1, L, L), g).reshape(-1, N)
                        if i < length - 1:
                            z = f.sum(1)
                            norm += torch.log(z)
                            # one start: the slice's W is the same for every message
                            f = f / z[:, None] * w[sg][(s0 + i + 1) % M if len(starts) > 1 else (starts[0] + i + 1) % M]
                    end = norm + torch.log(f.gather(1, i1[:, None])[:, 0])
                    which = torch.arange(k, k + i0.numel(), device="cuda") // len(starts)
                    logw[sg].index_add_(0, which, end)
        out.append(logw.reshape(-1))
    return torch.cat(out).cpu().numpy()


def _adjoint(case, seed):
    logz, dts, dvs = [], [], []
    for ((L, M, Nsig, U, dtau, cs), x, field), v in zip(_configuration(case, seed), _trained(case, seed)):
        N = L * L
        g, dg = _ring(L, dtau)
        w = torch.exp(v.double())
        dv = torch.zeros((2, M, N), dtype=torch.float64, device="cuda")
        lz = dt = 0.0
        most = max(1, int(2e9 / (N * M)))
        for sg in range(2):
            for k in range(0, Nsig, most):
                x0 = x[sg][k:k + most, 0]
                delta = torch.zeros((x0.numel(), N), dtype=torch.float64, device="cuda")
                delta.scatter_(1, x0[:, None], 1.0)
                kept, f, norm = [], delta, 0.0
                for l in range(M):
                    f = f * w[sg, l]
                    kept.append(f)
                    f = _propagate(f.view(-1, L, L), g).reshape(-1, N)
                    if l < M - 1:
                        z = f.sum(1, keepdim=True)
                        norm = norm + torch.log(z)
                        f = f / z
                lz += float((norm + torch.log(f.gather(1, x0[:, None]))).sum())
                b = delta
                for l in reversed(range(M)):
                    bl = b.view(-1, L, L)
                    h = _propagate(bl, g)
                    if L < 64:
                        d = dg @ bl @ g + g @ bl @ dg
                    else:  # dG/dt = dtau A G, A the lattice's adjacency
                        d = dtau * (h.roll(1, 1) + h.roll(-1, 1) + h.roll(1, 2) + h.roll(-1, 2))
                    h, d = h.reshape(-1, N), d.reshape(-1, N)
                    z = (kept[l] * h).sum(1, keepdim=True)
                    dv[sg, l] += (kept[l] * h / z).sum(0)
                    dt += float(((kept[l] * d).sum(1, keepdim=True) / z).sum())
                    b = h * w[sg, l]
                    b = b / b.sum(1, keepdim=True)
        logz.append(lz)
        dts.append(dt)
        dvs.append(dv.reshape(-1))
    return dict(logz=torch.tensor(logz, dtype=torch.float64), dv=torch.cat(dvs),
                dt=torch.tensor(sum(dts), dtype=torch.float64))


def exact(case, seed):
    """The log-weights and gradients; what a sweep draws has no such value, nor has a
    log-weight taken after a permutation update of the same sweep."""
    if case["kind"] == "adjoint":
        return _adjoint(case, seed)
    if case["kind"] == "local" or case["perm"]:
        return None
    return dict(logw=_filter_logw(case, seed))
