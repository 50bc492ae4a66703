"""Workloads of the walker-step library, for timing it: what a run of phaseless AFQMC has it do.

A case is a dict of plain values.  Its "kind" says which calls one pass makes:

  block  one block of a checkpointed run: restore the walkers, advance them `steps` steps on given
         fields (the energy measured every `measure` steps, re-orthonormalised every `qr` steps) and
         read the walkers back.  Outputs: the E_mix trace, the walkers and their weights.
  energy the mixed-estimator local energy of the current walkers.
  bp     the back-propagated one-body density matrix of a window of `steps` steps that have run.
  grad   local energy and log-overlap with their gradients (trial orbitals, Cholesky tensor).
  batch  `steps` steps of several uneven systems, then every system's walkers.

"ham" is the Hamiltonian's form (chol: real Cholesky vectors, cplx: complex ones, thc: tensor
hypercontraction), "trial" the trial (same: real, one determinant for both spins; uhf: real, one per
spin; complex; msd: `nd` non-orthogonal determinants), "prec" the walker set's precision.  The mixed
precision estimates carry about seven digits, so those cases keep their results in single precision,
as an archive of such a run does; FP64 results stay as they come.
"""
import math
import random

import numpy as np
import torch

from paper_2003_01831_gb300 import api, autograd, walkers

TAU = 0.005
MODES = {"phaseless": api.WEIGHT_PHASELESS, "free": api.WEIGHT_FREE, "local": api.WEIGHT_LOCAL}
MASK = (1 << 64) - 1


def _case(name, **kw):
    base = dict(kind="block", prec="fp64", ham="chol", trial="same", mode="phaseless", nd=1, nmu=0, nsys=0, steps=1,
                measure=1, qr=5, start=0, decay=20.0, fields="given")
    base.update(kw)
    if name is not None:
        base["name"] = name
    return base


def listed():
    return [
        # the small molecule of the parity workload: launches and latency are all there is
        _case("m24_fp64", M=24, nup=5, ndn=5, nchol=120, W=16, steps=5),
        # an open-shell molecule with a complex trial; no size is a multiple of anything
        _case("uhf90_fp64", M=90, nup=23, ndn=19, nchol=437, W=61, steps=2, trial="complex"),
        # the molecule-like workload in double precision, the reference run of a mixed one
        _case("m128_fp64", M=128, nup=32, ndn=32, nchol=640, W=512, qr=10),
        # the same molecule in tensor-hypercontraction form
        _case("thc128", M=128, nup=32, ndn=32, nchol=0, nmu=1024, W=64, ham="thc", qr=10),
        # a multi-determinant (non-orthogonal) trial
        _case("msd128", M=128, nup=32, ndn=32, nchol=640, W=32, trial="msd", nd=4, qr=10),
        # complex Cholesky vectors, as twisted boundary conditions give
        _case("cplx128", M=128, nup=32, ndn=32, nchol=640, W=48, ham="cplx", qr=10),
        # gradients for optimising a trial and a factorisation
        _case("grad128", kind="grad", M=128, nup=32, ndn=32, nchol=640, W=32),
        # the molecule-like workload in mixed precision, the energy at every step, one QR in the block
        _case("m128_mixed", prec="mixed", M=128, nup=32, ndn=32, nchol=640, W=512, steps=5),
        # equilibration: most steps only need the force bias; the energy at one step in five
        _case("m256_mixed", prec="mixed", M=256, nup=64, ndn=64, nchol=1280, W=256, steps=5, measure=5),
        # the throughput workload (solid-like), two steps with the energy at each and one QR
        _case("m512_mixed", prec="mixed", M=512, nup=128, ndn=128, nchol=2560, W=1024, steps=2, start=3,
              decay=200.0, fields="philox"),
        # observables that do not commute with H
        _case("bp256_mixed", kind="bp", prec="mixed", M=256, nup=64, ndn=64, nchol=1280, W=128, steps=2),
        # many small uneven problems at once
        _case("batch_mixed", kind="batch", prec="mixed", nsys=12, M=128, W=128, steps=2, fields="philox"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pad(n, m):
    return -(-n // m) * m


# A drawn case's cost, in flops with electrons padded as small blocks are, stays below these.
_MOST = {"fp64": 3.0e11, "mixed": 6.0e13}


def _cost(c):
    if c["kind"] == "batch":
        return sum(_cost(_case(None, prec="mixed", M=m, nup=n, ndn=n, nchol=k, W=w, steps=c["steps"]))
                   for m, n, k, w in _batch_dims(c))
    if c["prec"] == "mixed":
        d = dict(c, M=_pad(c["M"], 64), nup=_pad(c["nup"], 16), ndn=_pad(c["ndn"], 16))
    else:
        d = dict(c, nup=_pad(c["nup"], 32), ndn=_pad(c["ndn"], 32), M=_pad(c["M"], 32))
    return work(d)["flops"]


def draw(rng: random.Random):
    """One more case: a kind of run, and sizes over its whole range."""
    what = rng.choice(["fp64", "fp64", "uhf", "thc", "msd", "cplx", "grad", "mixed", "mixed", "mixed", "bp", "batch"])
    steps = rng.randint(1, 5)
    if what == "batch":
        c = _case(None, kind="batch", prec="mixed", nsys=rng.randint(2, 16), M=_log_int(rng, 48, 160),
                  W=_log_int(rng, 16, 160), steps=rng.randint(1, 2), fields="philox")
    elif what in ("mixed", "bp"):
        M = 64 * _log_int(rng, 1, 8)
        N = 8 * _log_int(rng, 1, min(16, M // 16))
        c = _case(None, prec="mixed", M=M, nup=N, ndn=N, nchol=8 * _log_int(rng, M // 8, 5 * M // 8),
                  W=_log_int(rng, 4, 1024 if M < 512 else 256), steps=steps, measure=rng.choice([1, 1, steps]),
                  start=rng.randint(0, 4), decay=rng.choice([20.0, 200.0]))
        if what == "bp":
            c.update(kind="bp", steps=rng.randint(1, 3), measure=1, start=0)
        elif rng.random() < 0.25:
            c.update(kind="energy", steps=1, measure=1)
    else:
        M = _log_int(rng, 12, 176)
        nup = _log_int(rng, 2, max(2, M // 3))
        c = _case(None, M=M, nup=nup, ndn=nup, nchol=_log_int(rng, M, 6 * M), W=_log_int(rng, 1, 512), steps=steps,
                  measure=rng.choice([1, 1, steps]), start=rng.randint(0, 4),
                  mode=rng.choice(["phaseless", "phaseless", "phaseless", "local", "free"]))
        if what == "uhf":
            c.update(ndn=max(1, nup - rng.randint(0, 3)), trial=rng.choice(["uhf", "complex"]))
        elif what == "thc":
            c.update(ham="thc", nmu=_log_int(rng, 4 * M, 9 * M), nchol=0)
        elif what == "msd":
            c.update(trial="msd", nd=rng.randint(2, 6))
        elif what == "cplx":
            c.update(ham="cplx", nchol=_log_int(rng, M, 5 * M))
        elif what == "grad":
            c.update(kind="grad", M=min(M, 128), nup=min(nup, 32), ndn=min(nup, 32), steps=1, measure=1,
                     mode="phaseless", trial=rng.choice(["same", "complex"]))
    while _cost(c) > _MOST[c["prec"]] and (c["W"] > 1 or c["steps"] > 1):
        if c["W"] > 1:
            c["W"] = c["W"] * 2 // 3
        else:
            c["steps"] -= 1
            c["measure"] = min(c["measure"], c["steps"])
    return c


# ------------------------------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _cnormal(g, *shape):
    return torch.complex(_normal(g, *shape), _normal(g, *shape))


def _one_body(g, M, band):
    if band:   # solid-like: a band of N(0, 0.2)
        h = 0.2 * _normal(g, M, M)
        i = torch.arange(M, device="cuda")
        h = torch.where((i[:, None] - i[None, :]).abs() <= 64, h, 0.0)
    else:      # molecule-like: diagonal U[-2, 2], off-diagonal N(0, 0.1)
        h = 0.1 * _normal(g, M, M)
        h.diagonal().copy_(4.0 * torch.rand(M, generator=g, device="cuda", dtype=torch.float64) - 2.0)
    return (torch.triu(h) + torch.triu(h, 1).mT).contiguous()


def _cholesky(g, M, nchol, decay):
    """Real symmetric vectors N(0, 1) x 0.5 exp(-n / decay) / sqrt(M)."""
    L = torch.empty(nchol, M, M, device="cuda", dtype=torch.float64)
    step = max(1, (1 << 26) // (M * M))
    for n in range(0, nchol, step):
        a = _normal(g, min(step, nchol - n), M, M)
        s = 0.5 / math.sqrt(M) * torch.exp(-torch.arange(n, n + a.shape[0], device="cuda", dtype=torch.float64) / decay)
        L[n:n + a.shape[0]] = (torch.triu(a) + torch.triu(a, 1).mT) * s[:, None, None]
    return L


def _inputs(c, seed):
    """What the program has in hand: a dict of tensors on the GPU, made from the seed alone."""
    g = _gen(seed)
    M, W, N = c["M"], c["W"], (c["nup"], c["ndn"])
    d = {"h": _one_body(g, M, c["decay"] > 100.0)}
    if c["ham"] == "thc":
        d["X"] = _normal(g, M, c["nmu"]) / math.sqrt(M)
        B = 0.5 / math.sqrt(c["nmu"]) * _normal(g, c["nmu"], c["nmu"])
        Mk = B @ B.mT
        d["Mk"] = (0.5 * (Mk + Mk.mT)).contiguous()
        nf = c["nmu"]
    elif c["ham"] == "cplx":
        n = torch.arange(c["nchol"], device="cuda", dtype=torch.float64)
        s = 0.35 / math.sqrt(M) * torch.exp(-n / c["decay"])
        d["L"] = (_cnormal(g, c["nchol"], M, M) * s[:, None, None]).contiguous()
        nf = 2 * c["nchol"]
    else:
        d["L"] = _cholesky(g, M, c["nchol"], c["decay"])
        nf = c["nchol"]
    # trial: the lowest orbitals of h, rotated for the unrestricted, complex and several-determinant ones
    v = torch.from_numpy(np.linalg.eigh(d["h"].cpu().numpy())[1]).cuda()
    low = [v[:, :n].to(torch.complex128).contiguous() for n in N]
    if c["trial"] == "uhf":
        low = [torch.linalg.qr((p + 0.1 / math.sqrt(M) * _normal(g, *p.shape)).real.cpu())[0].cuda().to(torch.complex128).contiguous()
               for p in low]
    elif c["trial"] == "complex":
        low = [torch.linalg.qr((p + 0.1 / math.sqrt(M) * _cnormal(g, *p.shape)).cpu())[0].cuda().contiguous() for p in low]
    if c["trial"] == "msd":
        d["Psi"] = [(p[None] + 0.3 / math.sqrt(M) * _cnormal(g, c["nd"], *p.shape)).contiguous() for p in low]
        d["coef"] = _cnormal(g, c["nd"])
    else:
        d["Psi"] = low
    # walkers as the phaseless walk spreads them around the trial, with weights around one
    amp = 0.5 / math.sqrt(M)
    near = [p[0] if c["trial"] == "msd" else p for p in d["Psi"]]
    d["Phi"] = torch.cat([(p[None] + amp * _cnormal(g, W, *p.shape)).reshape(W, -1) for p in near], dim=1).contiguous()
    d["w"] = torch.exp(0.2 * _normal(g, W))
    if c["mode"] == "free":
        d["w"] = d["w"].to(torch.complex128)
    d["dE"], d["dS"] = _cnormal(g, W), _cnormal(g, W)
    if c["fields"] == "given" and c["kind"] in ("block", "bp"):
        d["x"] = _normal(g, c["steps"], W, nf)
    d["seed"] = seed * 7919 + 1
    return d


def _batch_dims(c):
    """(M, N, Nchol, W) of the systems of a batch: sizes from a quarter of the largest up, N = M / 4, Nchol = 5 M."""
    r = random.Random(1003 + c["nsys"])
    out = []
    for _ in range(c["nsys"]):
        M = r.randint(max(8, c["M"] // 4), c["M"])
        out.append((M, max(1, M // 4), 5 * M, r.randint(max(1, c["W"] // 4), c["W"])))
    return out


def _batch_inputs(c, seed):
    out = []
    for s, (M, N, nchol, W) in enumerate(_batch_dims(c)):
        g = _gen(seed * 64 + s)
        h, L = _one_body(g, M, False), _cholesky(g, M, nchol, 20.0)
        v = np.linalg.eigh(h.cpu().numpy())[1]
        out.append((h, L, np.ascontiguousarray(v[:, :N].astype(np.complex128)), W))
    return out


class _State:
    """The handles and buffers that the program keeps."""

    ham = wk = None

    def __del__(self):
        try:
            if self.wk:
                api.afqmc_destroy_walkers(self.wk)
            if self.ham:
                api.afqmc_destroy_hamiltonian(self.ham)
        except Exception:
            pass


def _opts(c):
    o = api.afqmc_default_opts()
    o.precision = api.PREC_BF16X3 if c["prec"] == "mixed" else api.PREC_FP64
    o.k_qr = c["qr"]
    o.weight_mode = MODES[c["mode"]]
    return o


def prepare(case, seed):
    c = dict(case)
    s = _State()
    s.c = c
    if c["kind"] == "batch":
        systems = [(h.cpu().numpy(), L.cpu().numpy(), 0.0, P, P, W) for h, L, P, W in _batch_inputs(c, seed)]
        s.batch = walkers.Batch(systems, TAU, precision=api.PREC_BF16X3, k_qr=c["qr"])
        s.seed = seed
        s.out = [(torch.empty(W, M * 2 * N, device="cuda", dtype=torch.complex128),
                  torch.empty(W, device="cuda", dtype=torch.float64)) for M, N, _, W in _batch_dims(c)]
        s.trace = torch.empty(c["steps"], c["nsys"], device="cuda", dtype=torch.complex128)
        return s
    d = _inputs(c, seed)
    M, W = c["M"], c["W"]
    if c["kind"] == "grad":
        W0 = c["M"] * c["nup"]
        s.Psi = [p.clone().requires_grad_(True) for p in d["Psi"]]
        s.L = d["L"].requires_grad_(True)
        s.h, s.dE, s.dS = d["h"], d["dE"], d["dS"]
        s.Phi = [d["Phi"][:, :W0].reshape(W, M, -1).contiguous(), d["Phi"][:, W0:].reshape(W, M, -1).contiguous()]
        return s
    if c["ham"] == "thc":
        s.ham = api.afqmc_create_hamiltonian_thc(d["h"], d["X"], d["Mk"], 0.0, M, c["nmu"])
    elif c["ham"] == "cplx":
        s.ham = api.afqmc_create_hamiltonian_complex(d["h"], d["L"], 0.0, M, c["nchol"])
    else:
        s.ham = api.afqmc_create_hamiltonian(d["h"], d["L"], 0.0, M, c["nchol"])
    if c["trial"] == "msd":
        s.wk = api.afqmc_init_walkers_msd(s.ham, c["nd"], d["Psi"][0], d["Psi"][1], d["coef"], c["nup"], c["ndn"], W,
                                          d["Phi"], TAU, _opts(c))
    else:
        s.wk = api.afqmc_init_walkers(s.ham, d["Psi"][0], d["Psi"][1], c["nup"], c["ndn"], W, d["Phi"], TAU, _opts(c))
    s.Phi0, s.w0, s.seed = d["Phi"], d["w"], d["seed"]
    nf = api.afqmc_hamiltonian_info(s.ham)[1]
    s.x = d["x"][..., :nf].contiguous() if "x" in d else None
    if c["kind"] == "bp":
        api.afqmc_set_walkers(s.wk, s.Phi0, s.w0, 0)
        api.afqmc_bp_begin(s.wk, c["steps"])
        api.afqmc_step(s.wk, c["steps"], s.x, s.seed, 0, None)
        s.rdm = [torch.empty(M, M, device="cuda", dtype=torch.complex128) for _ in range(2)]
    elif c["kind"] == "energy":
        api.afqmc_set_walkers(s.wk, s.Phi0, s.w0, 0)
        s.E, s.logS = (torch.empty(W, device="cuda", dtype=torch.complex128) for _ in range(2))
        s.Emix = torch.empty(1, device="cuda", dtype=torch.complex128)
    else:
        s.Phi, s.w = torch.empty_like(s.Phi0), torch.empty_like(s.w0)
        s.trace = torch.empty(-(-c["steps"] // c["measure"]), device="cuda", dtype=torch.complex128)
    return s


def _kept(c, out):
    """Mixed-precision results are archived in single precision."""
    if c["prec"] != "mixed":
        return out
    return {k: v.to(torch.complex64 if v.is_complex() else torch.float32) for k, v in out.items()}


def run(s):
    c = s.c
    if c["kind"] == "block":
        api.afqmc_set_walkers(s.wk, s.Phi0, s.w0, c["start"])
        api.afqmc_step(s.wk, c["steps"], s.x, s.seed, c["measure"], s.trace)
        api.afqmc_get_walkers(s.wk, s.Phi, s.w)
        return _kept(c, {"E_mix": s.trace, "Phi": s.Phi, "w": s.w})
    if c["kind"] == "energy":
        api.afqmc_energy(s.wk, s.E, None, s.logS, s.Emix)
        return _kept(c, {"E_L": s.E, "E_mix": s.Emix, "logS": s.logS})
    if c["kind"] == "bp":
        api.afqmc_bp_rdm1(s.wk, s.rdm[0], s.rdm[1])
        return _kept(c, {"up": s.rdm[0], "dn": s.rdm[1]})
    if c["kind"] == "grad":
        E, logS = autograd.local_energy(s.Psi[0], s.Psi[1], s.L, s.h, 0.0, s.Phi[0], s.Phi[1])
        loss = (s.dE.conj() * E).real.sum() + (s.dS.conj() * logS).real.sum()
        gu, gd, gL = torch.autograd.grad(loss, (s.Psi[0], s.Psi[1], s.L))
        return {"E_L": E.detach(), "logS": logS.detach(), "dPsi_up": gu, "dPsi_dn": gd, "dL": gL}
    api.afqmc_batch_step(s.batch.b, c["steps"], s.seed, 1, s.trace)
    out = {"E_mix": s.trace}
    for k, (Phi, w) in enumerate(s.out):
        api.afqmc_batch_get_walkers(s.batch.b, k, Phi, w)
        out["Phi%d" % k], out["w%d" % k] = Phi, w
    return _kept(c, out)


def work(case):
    """Flops and compulsory bytes of one pass: a complex multiply-add counts 8, a real by complex one 4."""
    c = case
    if c["kind"] == "batch":
        parts = [work(_case(None, prec="mixed", M=m, nup=n, ndn=n, nchol=k, W=w, steps=c["steps"]))
                 for m, n, k, w in _batch_dims(c)]
        return {q: sum(p[q] for p in parts) for q in ("bytes", "flops")}
    M, W = c["M"], c["W"]
    Ns = (c["nup"], c["ndn"])
    K = 2 * c["nchol"] if c["ham"] == "cplx" else (c["nmu"] if c["ham"] == "thc" else c["nchol"])
    lc = 8.0 if c["ham"] == "cplx" else 4.0                                        # L times a complex operand
    ltc = 4.0 if c["ham"] != "cplx" and c["trial"] in ("same", "uhf") else 8.0      # Psi^+ L_n times Theta
    sum_n, sum_n2, sum_n3 = (sum(float(n) ** p for n in Ns) for p in (1, 2, 3))
    if c["ham"] == "thc":
        ham_b = 8.0 * (M * M + M * c["nmu"] + c["nmu"] ** 2)
        energy = 4.0 * W * sum_n * M * c["nmu"] + 8.0 * W * sum_n * c["nmu"] ** 2 + 8.0 * W * 2 * c["nmu"] ** 2
        bias = 4.0 * W * sum_n * M * c["nmu"] + 8.0 * W * sum_n * c["nmu"] + 4.0 * W * 2 * c["nmu"] * K
        hs = 4.0 * W * c["nmu"] * K + 4.0 * W * M * M * c["nmu"]
    else:
        ham_b = 8.0 * M * M + (16.0 if c["ham"] == "cplx" else 8.0) * K * M * M
        energy = c["nd"] * W * K * (ltc * sum_n2 * M + 8.0 * sum_n2)
        bias = c["nd"] * W * K * ltc * sum_n * M
        hs = lc * W * K * M * M
    over = c["nd"] * W * (8.0 * sum_n2 * M + 8.0 * sum_n3)                          # overlap, inverse
    theta = c["nd"] * W * 8.0 * sum_n2 * M
    prop = hs + W * sum_n * M * M * (6 * 8.0 + 2 * lc)
    phi_b = 16.0 * W * M * sum_n
    trial_b = 16.0 * c["nd"] * M * sum_n
    if c["kind"] == "energy":
        return {"flops": over + theta + energy, "bytes": ham_b + phi_b + trial_b + 32.0 * W}
    if c["kind"] == "bp":
        return {"flops": c["steps"] * prop + over + theta + 8.0 * W * M * M * sum_n,
                "bytes": ham_b + phi_b + trial_b + 32.0 * M * M + 16.0 * c["steps"] * W * K}
    if c["kind"] == "grad":
        # forward energy, then per vector U_n = Theta (c_n - T_n), L_n U_n, and the walker sum V_n Psi^+
        back = W * K * (ltc * sum_n2 * M + 8.0 * sum_n2 * M + 4.0 * sum_n * M * M + 8.0 * sum_n * M) + 8.0 * K * M * M * sum_n
        return {"flops": 2 * (over + theta) + energy + back,
                "bytes": 2 * ham_b + phi_b + 2 * trial_b + 64.0 * W}
    meas = -(-c["steps"] // c["measure"]) if c["mode"] != "local" else c["steps"]
    qr = sum(1 for k in range(c["steps"]) if c["qr"] and (c["start"] + k + 1) % c["qr"] == 0)
    flops = c["steps"] * (over + theta + prop) + meas * energy + (c["steps"] - meas) * bias + qr * 16.0 * W * sum_n2 * M
    x_b = 8.0 * c["steps"] * W * K if c["fields"] == "given" else 0.0
    return {"flops": flops, "bytes": ham_b + 2 * phi_b + trial_b + x_b + 16.0 * W}


# --------------------------------------------------------------------------- the same in 64 bits, plainly

def _logdet(S):
    sign, logabs = torch.linalg.slogdet(S)
    return torch.complex(logabs, torch.angle(sign))


def _measure(Psi, V, h, Phi, energy=True):
    """(E_L, <V_n>, log-overlap) of one determinant at the walkers Phi (per spin [W, M, N])."""
    E, t_sum, X_sum, logS = 0.0, 0.0, 0.0, 0.0
    for P, F in zip(Psi, Phi):
        S = P.mH @ F
        Th = F @ torch.linalg.inv(S)
        logS = logS + _logdet(S)
        E = E + torch.einsum("ak,wka->w", P.mH @ h.to(P.dtype), Th)
        n = P.shape[1]
        Lt = torch.matmul(P.mH, V.to(P.dtype)) if V.shape[0] * V.shape[1] ** 2 < 1 << 28 else \
            torch.cat([torch.matmul(P.mH, v.to(P.dtype)) for v in V.split(256)])
        rows = Lt.reshape(-1, Lt.shape[2])
        t, X = [], []
        for part in Th.split(max(1, (1 << 31) // (rows.shape[0] * n * 16))):
            T = torch.matmul(rows, part).reshape(part.shape[0], Lt.shape[0], n, n)
            t.append(T.diagonal(dim1=2, dim2=3).sum(-1))
            if energy:
                X.append((T * T.mT).sum((2, 3)))
        t_sum = t_sum + torch.cat(t)
        X_sum = X_sum + torch.cat(X) if energy else X_sum
    return (E + 0.5 * (t_sum * t_sum - X_sum).sum(1) if energy else None), t_sum, logS


def _trial_measure(c, d, V, Phi, energy=True):
    if c["trial"] != "msd":
        return _measure(d["Psi"], V, d["h"], Phi, energy)
    each = [_measure([p[i] for p in d["Psi"]], V, d["h"], Phi, energy) for i in range(c["nd"])]
    ls = torch.stack([torch.log(d["coef"][i].conj()) + e[2] for i, e in enumerate(each)])
    m = ls.real.max(0).values
    u = torch.exp(ls - m)
    Z = u.sum(0)
    u = u / Z
    E = sum(u[i] * e[0] for i, e in enumerate(each)) if energy else None
    return E, sum(u[i][:, None] * e[1] for i, e in enumerate(each)), torch.log(Z) + m


def _trial_energy(c, d, V):
    if c["trial"] != "msd":
        return _measure(d["Psi"], V, d["h"], [p[None] for p in d["Psi"]])[0][0].real
    Phi = [p for p in d["Psi"]]
    num = den = 0.0
    top, rows = None, []
    for i in range(c["nd"]):
        E, _, ls = _measure([p[i] for p in d["Psi"]], V, d["h"], Phi)
        rows.append((E, torch.log(d["coef"][i].conj()) + torch.log(d["coef"]) + ls))
    top = max(float(r[1].real.max()) for r in rows)
    for E, l in rows:
        f = torch.exp(l - top)
        num, den = num + (f * E).sum(), den + f.sum()
    return (num / den).real


def _vectors(c, d):
    if c["ham"] == "cplx":
        L = d["L"]
        V = torch.empty(2 * L.shape[0], *L.shape[1:], device="cuda", dtype=torch.complex128)
        V[0::2], V[1::2] = 0.5 * (L + L.mH), (L - L.mH) / 2j
        return V
    if c["ham"] == "thc":
        Mk = d["Mk"].cpu().numpy()
        n = Mk.shape[0]
        diag, cols = np.diag(Mk).copy(), np.zeros((n, n))
        stop, r = 1e-12 * diag.max(), 0
        while r < n:
            p = int(np.argmax(diag))
            if diag[p] <= stop:
                break
            cols[:, r] = (Mk[:, p] - cols[:, :r] @ cols[p, :r]) / math.sqrt(diag[p])
            diag -= cols[:, r] ** 2
            diag[p] = 0.0
            r += 1
        U = torch.from_numpy(cols[:, :r].copy()).cuda()
        return torch.einsum("im,mn,km->nik", d["X"], U, d["X"]).contiguous()
    return d["L"]


def _orthonormal(F):
    for _ in range(2):   # Cholesky QR, repeated: the Q with a positive diagonal R
        R = torch.linalg.cholesky(F.mH @ F, upper=True)
        F = torch.linalg.solve_triangular(R, F, upper=True, left=False)
    return F


def _philox(seed, step, W, n):
    """Philox4x32-10 normals [W, n]: counter (n / 4, walker, step, 0), Box-Muller."""
    q = -(-n // 4)
    m32 = np.uint64(0xFFFFFFFF)
    c0, c1 = np.meshgrid(np.arange(q, dtype=np.uint64), np.arange(W, dtype=np.uint64))
    c2, c3 = np.full_like(c0, step & 0xFFFFFFFF), np.zeros_like(c0)
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = c0 * np.uint64(0xD2511F53), c2 * np.uint64(0xCD9E8D57)
        c0, c1, c2, c3 = ((p1 >> np.uint64(32)) ^ c1 ^ np.uint64(k0), p1 & m32,
                          (p0 >> np.uint64(32)) ^ c3 ^ np.uint64(k1), p0 & m32)
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    u = [(v.astype(np.float64) + 0.5) * 2.0 ** -32 for v in (c0, c1, c2, c3)]
    x = np.empty((W, q, 4))
    for i in (0, 2):
        r = np.sqrt(-2.0 * np.log(u[i]))
        x[..., i], x[..., i + 1] = r * np.cos(2 * np.pi * u[i + 1]), r * np.sin(2 * np.pi * u[i + 1])
    return torch.from_numpy(x.reshape(W, 4 * q)[:, :n].copy()).cuda()


def _mm(a, V, part=512):
    """sum_n a[w, n] V[n]: [W, M, M]."""
    out = 0.0
    for k in range(0, V.shape[0], part):
        v = V[k:k + part]
        out = out + (a[:, k:k + part] @ v.reshape(v.shape[0], -1).to(a.dtype))
    return out.reshape(a.shape[0], V.shape[1], V.shape[2])


def _run64(c, d, V, Phi, w, fields, steps, start):
    """`steps` steps; returns the E_mix trace, the walkers, their weights and the shifted fields."""
    sq, ET = math.sqrt(TAU), _trial_energy(c, d, V)
    hp = d["h"].to(V.dtype) - 0.5 * sum(torch.einsum("nij,nkj->ik", v, v.conj()) for v in V.split(256))
    e, u = torch.linalg.eigh(hp)
    B = ((u * torch.exp(-0.5 * TAU * e)) @ u.mH).to(torch.complex128)
    trace, coefs = [], []
    for k in range(steps):
        meas = c["measure"] > 0 and k % c["measure"] == 0
        E, t, ls = _trial_measure(c, d, V, Phi, meas or c["mode"] == "local")
        if meas:
            trace.append((w * E).sum() / w.sum())
        xb = -1j * sq * t
        if c["mode"] != "free":
            mag = xb.abs()
            xb = torch.where(mag > 1.0, xb / mag, xb)
        x = fields(start + k)
        cf = x - xb
        coefs.append(cf)
        A = 1j * sq * _mm(cf, V)
        new = []
        for F in Phi:
            P = B @ F
            acc = P
            for j in range(1, 7):
                P = (A @ P) / j
                acc = acc + P
            new.append(B @ acc)
        del A
        ln = _trial_measure(c, d, V[:1], new, False)[2]
        dl = ln - ls
        ex = dl + (x * xb).sum(1) - 0.5 * (xb * xb).sum(1) + TAU * ET
        if c["mode"] == "free":
            w = w * torch.exp(ex)
        else:
            f = torch.exp(ex.real)
            if c["mode"] == "local":
                b = 2.0 / sq
                f = torch.exp(-TAU * (torch.minimum(torch.maximum(E.real, ET - b), ET + b) - ET))
            w = w * f * torch.clamp(torch.cos(dl.imag), min=0.0)
        Phi = new
        if c["qr"] and (start + k + 1) % c["qr"] == 0:
            Phi = [torch.where((w != 0)[:, None, None], _orthonormal(F), F) for F in Phi]
    return trace, Phi, w, coefs, B


def exact(case, seed):
    c = case
    if work(c)["flops"] * (6.0 if c["kind"] == "grad" else 1.0) > 1.2e13:
        return None   # minutes in 64 bits
    if c["kind"] == "batch":
        out, traces = {}, []
        for s, (h, L, P, W) in enumerate(_batch_inputs(c, seed)):
            sub = _case(None, M=h.shape[0], nup=P.shape[1], ndn=P.shape[1], nchol=L.shape[0], W=W, qr=c["qr"])
            key = (seed + s * api.SEED_STRIDE) & MASK
            Psi = [torch.from_numpy(P).cuda()] * 2
            F = [p[None].expand(W, -1, -1).contiguous() for p in Psi]
            w = torch.ones(W, device="cuda", dtype=torch.float64)
            tr, F, w, _, _ = _run64(sub, {"h": h, "Psi": Psi}, L, F, w,
                                    lambda k: _philox(key, k, W, L.shape[0]), c["steps"], 0)
            traces.append(torch.stack(tr))
            out["Phi%d" % s] = torch.cat([f.reshape(W, -1) for f in F], dim=1)
            out["w%d" % s] = w
        out["E_mix"] = torch.stack(traces, dim=1)
        return out
    d = _inputs(c, seed)
    M, W = c["M"], c["W"]
    at = M * c["nup"]
    Phi = [d["Phi"][:, :at].reshape(W, M, -1), d["Phi"][:, at:].reshape(W, M, -1)]
    if c["kind"] == "grad":
        leaf = [p.clone().requires_grad_(True) for p in d["Psi"]]
        L = d["L"].clone().requires_grad_(True)
        Es, Ss, g = [], [], None
        for k in range(0, W, 4):   # a few walkers at a time
            E, _, ls = _measure(leaf, L, d["h"], [F[k:k + 4] for F in Phi])
            ls = torch.complex(ls.real, torch.atan2(torch.sin(ls.imag), torch.cos(ls.imag)))
            loss = (d["dE"][k:k + 4].conj() * E).real.sum() + (d["dS"][k:k + 4].conj() * ls).real.sum()
            new = torch.autograd.grad(loss, (leaf[0], leaf[1], L))
            g = new if g is None else [a + b for a, b in zip(g, new)]
            Es.append(E.detach())
            Ss.append(ls.detach())
        return {"E_L": torch.cat(Es), "logS": torch.cat(Ss), "dPsi_up": g[0], "dPsi_dn": g[1], "dL": g[2]}
    V = _vectors(c, d)
    if c["kind"] == "energy":
        E, _, ls = _trial_measure(c, d, V, Phi)
        ls = torch.complex(ls.real, torch.atan2(torch.sin(ls.imag), torch.cos(ls.imag)))
        return {"E_L": E, "E_mix": ((d["w"] * E).sum() / d["w"].sum()).reshape(1), "logS": ls}
    if c["fields"] == "given":
        fields = lambda k: d["x"][k - c["start"]][:, :V.shape[0]]
    else:
        fields = lambda k: _philox(d["seed"] & MASK, k, W, V.shape[0])
    trace, F, w, coefs, B = _run64(dict(c, measure=0) if c["kind"] == "bp" else c, d, V, Phi, d["w"], fields,
                                   c["steps"], c["start"])
    if c["kind"] == "bp":
        out = []
        for s in range(2):
            Q = d["Psi"][s][None].expand(W, -1, -1)
            for cf in reversed(coefs):
                A = (1j * math.sqrt(TAU) * _mm(cf, V)).mH
                P = B.mH @ Q
                acc = P
                for j in range(1, 7):
                    P = (A @ P) / j
                    acc = acc + P
                Q = B.mH @ acc
            Th = Phi[s] @ torch.linalg.inv(Q.mH @ Phi[s])
            out.append(((w[:, None, None] * Th) @ Q.mH).sum(0).mT / w.sum())
        return {"up": out[0], "dn": out[1]}
    return {"E_mix": torch.stack(trace), "Phi": torch.cat([f.reshape(W, -1) for f in F], dim=1), "w": w}
