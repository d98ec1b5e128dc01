"""Workloads of the two-site DMRG library, each one pass through its public entry points.

A case is a dict of plain values; ``kind`` says which call it stands for:

* ``sigma``       one H_eff.psi on device vectors at the central sites (the call a user's own
                  eigensolver makes), in one of the precisions of gbdmrg_set_precision;
* ``step``        one two-site update at the central sites: W-contracted operators, work
                  lists, diagonal, a fixed number of Davidson iterations, decimation and the
                  environment update (gbdmrg_step);
* ``run``         whole sweeps of a small problem from a random MPS (gbdmrg_run);
* ``batch``       sigma vectors of several independent problems in one launch per stage,
                  replayed from a CUDA graph (gbdmrg_batch_sigma);
* ``mlp_train``   training of the preconditioner network on device-resident pairs
                  (gbdmrg_mlp_train);
* ``mlp_grad``    its loss and gradient over a set of pairs (gbdmrg_mlp_loss_grad);
* ``mlp_forward`` the network applied to every element of a residual (gbdmrg_mlp_forward,
                  inference numerics).

Integrals, matrix product states, vectors, pairs and network parameters are all made from the
seed (paper_1605_02611_gb300.synth gives the integrals and the bond sectors).
"""
import ctypes
import math
import tempfile

import numpy as np
import torch

import paper_1605_02611_gb300 as G
from paper_1605_02611_gb300 import synth

HIDDEN, NFEAT = 256, 5


# ------------------------------------------------------------------ cases

def listed():
    return [
        # the exact benchmark problem (K=8, N=8, full bond dimension) on the FP64 path: a call
        # whose blocks are small, so that latency and padding count
        dict(name="sigma_f64_k8_m256", kind="sigma", K=8, N=8, two_sz=0, M=256, precision=0),
        # the FP64 path in the M ramp of the K=24 problem
        dict(name="sigma_f64_k24_m256", kind="sigma", K=24, N=24, two_sz=0, M=256, precision=0),
        # early sweeps of a tensor-core run, odd electron number: small ragged sectors
        dict(name="sigma_bf16x3_k10_m150", kind="sigma", K=10, N=9, two_sz=1, M=150, precision=5),
        # the K=24, M=512 problem on the default tensor-core path (three slices)
        dict(name="sigma_bf16x3_k24_m512", kind="sigma", K=24, N=24, two_sz=0, M=512, precision=5),
        # the same path in one BF16 pass at the size of the preconditioner workload
        dict(name="sigma_bf16_k32_m1024", kind="sigma", K=32, N=32, two_sz=0, M=1024, precision=4),
        # the K=40 problem of the headline on its way from M=1000 to 2000 (at M=2000 its work
        # lists alone take about 90 GB, so that three of them would not fit the device)
        dict(name="sigma_bf16x3_k40_m1200", kind="sigma", K=40, N=40, two_sz=0, M=1200, precision=5),
        # a two-site update entirely in FP64
        dict(name="step_f64_k16_m128", kind="step", K=16, N=16, two_sz=0, M=128, precision=0, env=0, iters=8),
        # a two-site update as the benchmark does it: three slices, exactly split environments
        dict(name="step_mixed_k24_m512", kind="step", K=24, N=24, two_sz=0, M=512, precision=5, env=3, iters=8),
        # a whole small calculation: launches, synchronisations and host planning count
        dict(name="run_f64_k6_m64", kind="run", K=6, N=6, two_sz=0, M=64, sweeps=2),
        # several problems of different sizes at once
        dict(name="batch_bf16x3_8", kind="batch", problems=8, kmin=12, kmax=20, mmin=64, mmax=256, precision=2),
        # training on collected pairs in minibatches of 4096
        dict(name="mlp_train_16384", kind="mlp_train", n=16384, batch=4096, epochs=1),
        # the network over all elements of a residual (about those of K=24, M=512)
        dict(name="mlp_forward_200000", kind="mlp_forward", n=200000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sigma_f64", "sigma_tc", "sigma_tc", "step_f64", "step_mixed", "run", "batch", "mlp_train",
                       "mlp_grad", "mlp_forward"])
    if kind in ("sigma_f64", "sigma_tc", "step_f64", "step_mixed"):
        top_k, top_m = {"sigma_f64": (24, 400), "sigma_tc": (32, 1000), "step_f64": (16, 160),
                        "step_mixed": (24, 512)}[kind]
        K = rng.randint(6, top_k)
        N = K + rng.randint(-2, 2)
        two_sz = N % 2 if rng.random() < 0.7 else N % 2 + 2
        case = dict(K=K, N=N, two_sz=two_sz, M=_log_int(rng, 24, top_m))
        if kind == "sigma_f64":
            return dict(kind="sigma", precision=0, **case)
        if kind == "sigma_tc":
            return dict(kind="sigma", precision=rng.choice([4, 5, 5, 6]), **case)
        if kind == "step_f64":
            return dict(kind="step", precision=0, env=0, iters=rng.randint(4, 10), **case)
        return dict(kind="step", precision=5, env=3, iters=rng.randint(4, 10), **case)
    if kind == "run":
        K = rng.randint(4, 7)
        return dict(kind="run", K=K, N=K, two_sz=K % 2, M=rng.randint(12, 64), sweeps=rng.randint(1, 2))
    if kind == "batch":
        kmin = rng.randint(8, 14)
        return dict(kind="batch", problems=rng.randint(2, 10), kmin=kmin, kmax=kmin + rng.randint(0, 6),
                    mmin=rng.randint(16, 64), mmax=rng.randint(64, 256), precision=rng.choice([1, 2, 3]))
    if kind == "mlp_train":
        batch = _log_int(rng, 500, 8192)
        return dict(kind="mlp_train", n=batch * rng.randint(1, 4) + rng.randint(-200, 200), batch=batch, epochs=1)
    if kind == "mlp_grad":
        return dict(kind="mlp_grad", n=_log_int(rng, 1000, 200000))
    return dict(kind="mlp_forward", n=_log_int(rng, 1000, 500000))


# ------------------------------------------------------------------ inputs

def _integrals(K, seed):
    # the problem statement's spread of the off-diagonal one-electron integrals
    return synth.integrals(K, seed, 0.05 if K >= 40 else 0.1)


def _isometric_mps(bonds, center, rng):
    """Random MPS in mixed-canonical form around sites (center, center + 1), as sweeps leave it:
    isometric blocks per bond sector (Q factors of Gaussian matrices), Gaussian centre tensors."""
    tensors = []
    for k in range(len(bonds) - 1):
        L, R = bonds[k], bonds[k + 1]
        A = np.zeros((L.total, 4, R.total))
        loff = np.cumsum([0] + list(L.dim))
        roff = np.cumsum([0] + list(R.dim))
        lsec = {q: (int(loff[i]), L.dim[i]) for i, q in enumerate(L.qn)}
        rsec = {q: (int(roff[i]), R.dim[i]) for i, q in enumerate(R.qn)}
        left = k < center
        for (qa, qb), (off, d) in (rsec if left else lsec).items():
            parts = []  # (n, offset, size) of the sectors that meet this one
            for n, (a, b) in enumerate(synth.LOCAL_QN):
                sec = lsec.get((qa - a, qb - b)) if left else rsec.get((qa + a, qb + b))
                if sec:
                    parts.append((n, sec[0], sec[1]))
            rows = sum(p[2] for p in parts)
            if rows == 0:
                continue
            X = rng.normal(size=(rows, d))
            if not center <= k <= center + 1:
                X, _ = np.linalg.qr(X)
            r0 = 0
            for n, o, m in parts:
                if left:
                    A[o:o + m, n, off:off + d] = X[r0:r0 + m]
                else:
                    A[off:off + d, n, o:o + m] = X[r0:r0 + m].T
                r0 += m
        tensors.append(A)
    return tensors


class _Problem:
    """One problem at its central sites: a context with its environments and work lists, and
    device vectors."""

    def __init__(self, K, N, two_sz, M, precision, seed, stream, env=3, keep=False):
        self.K, self.N, self.two_sz = K, N, two_sz
        self.k = K // 2 - 1
        self.h, self.eri = _integrals(K, seed)
        rng = np.random.default_rng(seed + 1)
        Na, Nb = (N + two_sz) // 2, (N - two_sz) // 2
        self.bonds = synth.bond_sectors(K, Na, Nb, M, 1.0)
        tensors = _isometric_mps(self.bonds, self.k, rng)
        self.ctx = G.Context(self.h, self.eri, N, two_sz, stream=stream.cuda_stream)
        self.ctx.set_precision(precision)
        self.ctx.set_env_precision(env)
        if keep:
            self.ctx.keep_host_plans(True)
        self.ctx.set_mps(tensors, [b.labels() for b in self.bonds])
        self.ctx.prepare(self.k)
        x = rng.normal(size=self.ctx.nnz)
        self.psi = x / np.linalg.norm(x)
        self.x = torch.tensor(self.psi, device="cuda")
        self.y = torch.empty_like(self.x)


def _network(seed):
    """Parameters of a partly trained network and pairs as Davidson leaves them: unit-RMS
    residual elements with heavy tails, logarithmic diagonal shifts, corrections near the
    diagonal one."""
    rng = np.random.default_rng(seed)
    p = np.concatenate([rng.normal(0, 1 / math.sqrt(NFEAT), HIDDEN * NFEAT), rng.normal(0, 0.05, HIDDEN),
                        rng.normal(0, 1 / math.sqrt(HIDDEN), HIDDEN * HIDDEN), rng.normal(0, 0.05, HIDDEN),
                        rng.normal(0, 0.02, HIDDEN), [0.01]])
    return p.astype(np.float32)


def _pairs(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    delta = torch.exp(torch.randn(n, generator=g, device="cuda") * 1.2)
    r = torch.randn(n, generator=g, device="cuda") * torch.exp(0.7 * torch.randn(n, generator=g, device="cuda"))
    F = torch.stack([r, torch.asinh(delta), delta / (delta * delta + 0.01),
                     torch.asinh(r.abs() * 0.5 + 0.5), torch.asinh(delta * 0.8 + 0.3)], 1).contiguous()
    P = (-r / delta).clamp(-100, 100)
    T = (P * (1 + 0.3 * torch.tanh(F[:, 1] - 1)) + 0.1 * torch.randn(n, generator=g, device="cuda")).clamp(-100, 100)
    return F, P, T


def _batch_sizes(case):
    n = case["problems"]
    at = [i / max(1, n - 1) for i in range(n)]
    return [(round(case["kmin"] + f * (case["kmax"] - case["kmin"])),
             round(case["mmin"] * (case["mmax"] / case["mmin"]) ** ((0.37 + 1.618 * i) % 1.0)))
            for i, f in enumerate(at)]


def prepare(case, seed):
    s = dict(case)
    kind = case["kind"]
    if kind in ("sigma", "step", "batch"):
        s["stream"] = torch.cuda.Stream()
    if kind == "sigma":
        # the environments of a sigma case are built on the tensor cores (exactly split
        # operands, FP64 level), which is the quicker way to the same operators
        s["p"] = _Problem(case["K"], case["N"], case["two_sz"], case["M"], case["precision"], seed, s["stream"],
                          env=0 if case["K"] <= 8 else 3)
    elif kind == "step":
        s["p"] = p = _Problem(case["K"], case["N"], case["two_sz"], case["M"], 0, seed, s["stream"], env=case["env"])
        # a solver without a guess starts from the unit vector of the lowest diagonal element
        p.x.zero_()
        p.x[int(np.argmin(p.ctx.diag()))] = 1.0
        if case["precision"]:
            p.ctx.set_precision(case["precision"])
            p.ctx.plan(p.k)
    elif kind == "batch":
        s["ps"] = [_Problem(K, K, K % 2, M, case["precision"], seed + 100 * i, s["stream"], keep=True)
                   for i, (K, M) in enumerate(_batch_sizes(case))]
        torch.cuda.synchronize()
        s["batch"] = G.Batch([p.ctx for p in s["ps"]])
        s["xs"] = [p.x.data_ptr() for p in s["ps"]]
        s["ys"] = [p.y.data_ptr() for p in s["ps"]]
    elif kind == "run":
        K, N = case["K"], case["N"]
        bonds, tensors = synth.random_mps(K, N, case["two_sz"], case["M"], seed + 1)
        s["ctx"] = G.Context(*_integrals(K, seed), N, case["two_sz"])
        s["ctx"].set_mps(tensors, [b.labels() for b in bonds])
        s["file"] = tempfile.NamedTemporaryFile()  # the start of every pass, as a calculation resumes
        s["ctx"].save(s["file"].name)
    else:
        s["params"] = _network(seed)
        s["F"], s["P"], s["T"] = _pairs(case["n"], seed)
        s["net"] = G.Mlp(seed)
        s["net"].set_params(s["params"])
        s["g"] = torch.empty(case["n"], device="cuda")
    torch.cuda.synchronize()
    return s


# ------------------------------------------------------------------ passes

def _fp32_values(y, precision):
    """A tensor-core sigma holds the FP32 sums of the accumulators, widened; a program that keeps
    it keeps those.  The FP64 path's is FP64."""
    return y.to(torch.float32) if precision > 0 else y


def run(s):
    kind = s["kind"]
    if kind == "sigma":
        p = s["p"]
        with torch.cuda.stream(s["stream"]):
            p.ctx.sigma_device(p.x.data_ptr(), p.y.data_ptr())
            return _fp32_values(p.y, s["precision"])
    if kind == "step":
        p = s["p"]
        with torch.cuda.stream(s["stream"]):
            # the site tensors are not returned: their gauge (the signs of the eigenvectors kept
            # by the decimation) is free.  The vector of a tensor-core step carries FP32 accuracy.
            e, d, _, _ = p.ctx.step(p.k, 0, s["M"], 1e-14, s["iters"], psi_in=p.x.data_ptr(),
                                    want_psi=p.y.data_ptr(), on_device=True)
            y = _fp32_values(p.y, s["precision"])
        return {"energy": _fp32_scalar(e, d, s["precision"]), "psi": y}
    if kind == "batch":
        with torch.cuda.stream(s["stream"]):
            s["batch"].sigma(s["xs"], s["ys"], True)
            return [_fp32_values(p.y, s["precision"]) for p in s["ps"]]
    if kind == "run":
        s["ctx"].load(s["file"].name)
        e = s["ctx"].run([s["M"]] * s["sweeps"], 1e-8, 60)["energy"]
        return {"before": e[:-1], "last": e[-1:]}
    net, n = s["net"], s["n"]
    lib, ptr = net.lib, lambda t: ctypes.c_void_p(t.data_ptr())
    if kind == "mlp_forward":
        net._check(lib.gbdmrg_mlp_forward(net.h, ptr(s["F"]), n, ptr(s["g"]), 1, 1), "forward")
        return s["g"]
    loss = ctypes.c_double()
    if kind == "mlp_grad":
        grad = np.zeros(net.nparams, dtype=np.float32)
        net._check(lib.gbdmrg_mlp_loss_grad(net.h, ptr(s["F"]), ptr(s["P"]), ptr(s["T"]), n, 1,
                                            grad.ctypes.data_as(ctypes.POINTER(ctypes.c_float)),
                                            ctypes.byref(loss)), "loss_grad")
        return {"loss": np.array([loss.value], dtype=np.float32), "grad": grad}
    net.set_params(s["params"])
    net._check(lib.gbdmrg_mlp_train(net.h, ptr(s["F"]), ptr(s["P"]), ptr(s["T"]), n, 1, s["epochs"], s["batch"], 1e-3,
                                    17, ctypes.byref(loss), None), "train")
    return {"loss": np.array([loss.value], dtype=np.float32), "params": net.get_params()}


def _fp32_scalar(e, d, precision):
    return np.array([e, d], dtype=np.float32 if precision > 0 else np.float64)


# ------------------------------------------------------------------ work

def _sigma_flops(K, N, two_sz, bonds, k):
    h, eri = _integrals(K, 1)
    return G.sigma_flops_host(h, eri, N, two_sz, k, bonds[k].labels(), bonds[k + 2].labels())


def _op_nnz(bond, da, db):
    dims = dict(zip(bond.qn, bond.dim))
    return sum(d * dims.get((a + da, b + db), 0) for (a, b), d in dims.items())


def _env_values(K, b, bond):
    """Values of the renormalised operators of bond b: identity and Hamiltonian, one-index
    operators (normal and complementary, 2 per orbital and spin) and the two-index operators of
    the shorter side."""
    n = min(b, K - b)
    total = 2 * _op_nnz(bond, 0, 0)
    for q in ((1, 0), (0, 1), (-1, 0), (0, -1)):
        total += K * _op_nnz(bond, *q)
    for s in (1, -1):
        total += n * (n - 1) // 2 * (_op_nnz(bond, 2 * s, 0) + _op_nnz(bond, 0, 2 * s)) + n * n * _op_nnz(bond, s, s)
        total += n * n * _op_nnz(bond, s, -s)
    return total + 2 * n * n * _op_nnz(bond, 0, 0)


def _psi_nnz(bl, br):
    dims = dict(zip(br.qn, br.dim))
    return sum(d * dims.get((a + x + u, b + y + v), 0) for (a, b), d in zip(bl.qn, bl.dim)
               for x, y in synth.LOCAL_QN for u, v in synth.LOCAL_QN)


def _problem_work(K, N, two_sz, M, sigmas):
    bonds = synth.bond_sectors(K, (N + two_sz) // 2, (N - two_sz) // 2, M, 1.0)
    k = K // 2 - 1
    env = 8 * (_env_values(K, k, bonds[k]) + _env_values(K, k + 2, bonds[k + 2]))
    return (16 * _psi_nnz(bonds[k], bonds[k + 2]) + env, sigmas * _sigma_flops(K, N, two_sz, bonds, k),
            8 * _env_values(K, k + 1, bonds[k + 1]))


def work(case):
    kind = case["kind"]
    if kind == "sigma":
        b, f, _ = _problem_work(case["K"], case["N"], case["two_sz"], case["M"], 1)
        return {"bytes": b, "flops": f}
    if kind == "step":
        # the new environment is written; the sigma vectors of the iterations
        b, f, e = _problem_work(case["K"], case["N"], case["two_sz"], case["M"], case["iters"] + 1)
        return {"bytes": b + e, "flops": f}
    if kind == "batch":
        w = [_problem_work(K, K, K % 2, M, 1) for K, M in _batch_sizes(case)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    if kind == "run":
        # at least two sigma vectors at every step of a sweep
        K, N, two_sz = case["K"], case["N"], case["two_sz"]
        bonds = synth.bond_sectors(K, (N + two_sz) // 2, (N - two_sz) // 2, case["M"])
        f = sum(_sigma_flops(K, N, two_sz, bonds, k) for k in list(range(K - 2)) + list(range(K - 2, 0, -1)))
        b = sum(16 * _psi_nnz(bonds[k], bonds[k + 2]) for k in list(range(K - 2)) + list(range(K - 2, 0, -1)))
        return {"bytes": 2 * case["sweeps"] * b, "flops": 2 * case["sweeps"] * f}
    rows = case["n"]
    if kind == "mlp_train":
        rows = -(-case["n"] // case["batch"]) * case["batch"] * case["epochs"]
    per = 2 * (NFEAT * HIDDEN + HIDDEN * HIDDEN + HIDDEN)
    if kind == "mlp_forward":
        return {"bytes": 4 * (NFEAT + 1) * rows, "flops": per * rows}
    return {"bytes": 4 * (NFEAT + 2) * rows + 8 * (HIDDEN * HIDDEN + 7 * HIDDEN + 1), "flops": 3 * per * rows}


# ------------------------------------------------------------------ 64-bit values

class _Fock:
    """H of the integrals on the 4^K occupation vectors of K spatial orbitals (site 0 the most
    significant digit n = n_up + 2 n_dn, Jordan-Wigner order 0up, 0dn, 1up, ...), FP64."""

    def __init__(self, h, eri):
        self.K = K = h.shape[0]
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.eri = torch.tensor(eri.reshape(K * K, K * K), device=dev)
        self.h = torch.tensor((h - 0.5 * np.einsum("prrq->pq", eri)).reshape(-1), device=dev)
        idx = torch.arange(4 ** K, device=dev)
        bit = lambda p, s: 2 * (K - 1 - p) + s  # noqa: E731
        self.e = []  # per (p, q), both spins: (from, to, sign) of a+_p a_q
        for p in range(K):
            for q in range(K):
                ops = []
                for s in (0, 1):
                    src = idx[(idx >> bit(q, s)) & 1 == 1]
                    cut, sg = src ^ (1 << bit(q, s)), self._before(src, q, s)
                    free = (cut >> bit(p, s)) & 1 == 0
                    src, cut, sg = src[free], cut[free], sg[free]
                    ops.append((src, cut | (1 << bit(p, s)), (1 - 2 * ((sg + self._before(cut, p, s)) & 1)).double()))
                self.e.append([torch.cat(t) for t in zip(*ops)])

    def _before(self, x, p, s):
        """Electrons in the spin orbitals that come before (p, s)."""
        c = torch.zeros_like(x)
        for b in range(2 * (self.K - p), 2 * self.K):
            c += (x >> b) & 1
        return c + ((x >> (2 * (self.K - 1 - p))) & 1 if s else 0)

    def one(self, j, v):
        src, dst, sg = self.e[j]
        return torch.zeros_like(v).index_add_(0, dst, sg * v[src])

    def apply(self, v):
        w = torch.stack([self.one(j, v) for j in range(self.K ** 2)])
        u = 0.5 * (self.eri @ w) + self.h[:, None] * v[None]
        return sum(self.one(j, u[j]) for j in range(self.K ** 2))

    def lowest(self, Na, Nb):
        """Lowest eigenvalue with Na up and Nb down electrons (Lanczos, full orthogonalisation)."""
        idx = torch.arange(4 ** self.K, device=self.h.device)
        na, nb = torch.zeros_like(idx), torch.zeros_like(idx)
        for p in range(self.K):
            na += (idx >> (2 * p)) & 1
            nb += (idx >> (2 * p + 1)) & 1
        sector = ((na == Na) & (nb == Nb)).double()
        g = torch.Generator(device=self.h.device).manual_seed(3)
        v = sector * torch.randn(len(idx), generator=g, device=self.h.device, dtype=torch.float64)
        V, a, b = [v / v.norm()], [], []
        for _ in range(min(200, int(sector.sum()))):
            w = self.apply(V[-1])
            a.append(float(w @ V[-1]))
            Q = torch.stack(V)
            for _ in range(2):
                w = w - Q.T @ (Q @ w)
            n = float(w.norm())
            if n < 1e-9:
                break
            b.append(n)
            V.append(w / n)
        m = len(a)
        return float(np.linalg.eigvalsh(np.diag(a) + np.diag(b[:m - 1], 1) + np.diag(b[:m - 1], -1))[0])


def _sigma_exact(case, seed):
    """P^T H P psi with the bases of both sides as explicit occupation vectors."""
    K, M = case["K"], case["M"]
    h, eri = _integrals(K, seed)
    rng = np.random.default_rng(seed + 1)
    bonds = synth.bond_sectors(K, (case["N"] + case["two_sz"]) // 2, (case["N"] - case["two_sz"]) // 2, M, 1.0)
    k = K // 2 - 1
    A = _isometric_mps(bonds, k, rng)
    Lb, Rb = bonds[k], bonds[k + 2]
    lo, ro = np.cumsum([0] + list(Lb.dim)), np.cumsum([0] + list(Rb.dim))
    rsec = {q: j for j, q in enumerate(Rb.qn)}
    blocks = []  # the packed layout: left sector, n1, n2, each block row-major
    for i, (a, b) in enumerate(Lb.qn):
        for n1, (x, y) in enumerate(synth.LOCAL_QN):
            for n2, (u, v) in enumerate(synth.LOCAL_QN):
                j = rsec.get((a + x + u, b + y + v))
                if j is not None:
                    blocks.append((slice(lo[i], lo[i + 1]), n1, n2, slice(ro[j], ro[j + 1])))
    psi = np.zeros((Lb.total, 4, 4, Rb.total))
    sizes = [(b[0].stop - b[0].start, b[3].stop - b[3].start) for b in blocks]
    x = rng.normal(size=sum(m * n for m, n in sizes))
    x /= np.linalg.norm(x)
    o = 0
    for (l, n1, n2, r), (m, n) in zip(blocks, sizes):
        psi[l, n1, n2, r] = x[o:o + m * n].reshape(m, n)
        o += m * n
    left = np.ones((1, 1))
    for t in A[:k]:
        left = np.einsum("xl,lnr->xnr", left, t, optimize=True).reshape(-1, t.shape[2])
    right = np.ones((1, 1))
    for t in reversed(A[k + 2:]):
        right = np.einsum("lnr,rx->lnx", t, right, optimize=True).reshape(t.shape[0], -1)
    F = _Fock(h, eri)
    dev = F.h.device
    left, right, psi = (torch.tensor(t, device=dev) for t in (left, right, psi))
    v = torch.einsum("xl,lpqr,ry->xpqy", left, psi, right).reshape(-1)
    s = torch.einsum("xl,xpqy,ry->lpqr", left, F.apply(v).reshape(left.shape[0], 4, 4, right.shape[1]), right)
    return torch.cat([s[l, n1, n2, r].reshape(-1) for l, n1, n2, r in blocks])


def _bf16(t):
    return t.to(torch.float32).to(torch.bfloat16).double()


def _unpack(p):
    o = [0]
    for n in (HIDDEN * NFEAT, HIDDEN, HIDDEN * HIDDEN, HIDDEN, HIDDEN, 1):
        o.append(o[-1] + n)
    w = [p[a:b] for a, b in zip(o, o[1:])]
    return w[0].reshape(HIDDEN, NFEAT), w[1], w[2].reshape(HIDDEN, HIDDEN), w[3], w[4], w[5]


def _loss_grad(p, F, P, T):
    """Loss mean(((1 + g) P - T)^2) and its gradient, weights rounded to BF16 (straight through)."""
    q = [t.detach().clone() for t in _unpack(p)]
    for i in (0, 2, 4):
        q[i] = _bf16(q[i])
    q = [t.requires_grad_(True) for t in q]
    loss = 0.0
    for a in range(0, len(F), 1 << 16):
        f = F[a:a + (1 << 16)].double()
        gelu = torch.nn.functional.gelu
        g = gelu(gelu(f @ q[0].T + q[1]) @ q[2].T + q[3]) @ q[4] + q[5]
        part = (((1 + g) * P[a:a + (1 << 16)].double() - T[a:a + (1 << 16)].double()) ** 2).sum() / len(F)
        part.backward()
        loss += float(part)
    return loss, torch.cat([t.grad.reshape(-1) for t in q])


def _splitmix(x):
    with np.errstate(over="ignore"):
        z = np.asarray(x, dtype=np.uint64) + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def exact(case, seed):
    kind = case["kind"]
    if kind == "sigma":
        return _sigma_exact(case, seed) if case["K"] <= 10 else None
    if kind == "run":
        # the sweeps are exact once every bond holds all its states
        if case["M"] < 4 ** (case["K"] // 2) or case["sweeps"] < 2:
            return None
        h, eri = _integrals(case["K"], seed)
        e = _Fock(h, eri).lowest((case["N"] + case["two_sz"]) // 2, (case["N"] - case["two_sz"]) // 2)
        return {"before": None, "last": np.array([e])}
    if kind in ("step", "batch"):
        return None
    p = torch.tensor(_network(seed), device="cuda").double()
    F, P, T = _pairs(case["n"], seed)
    if kind == "mlp_forward":
        w1, b1, w2, b2, w3, b3 = _unpack(p)
        gelu, out = torch.nn.functional.gelu, []
        for a in range(0, len(F), 1 << 16):
            h1 = _bf16(gelu(F[a:a + (1 << 16)].double() @ _bf16(w1).T + b1))
            out.append(gelu(h1 @ _bf16(w2).T + b2) @ _bf16(w3) + b3)
        return torch.cat(out)
    if kind == "mlp_grad":
        loss, grad = _loss_grad(p, F, P, T)
        return {"loss": np.array([loss]), "grad": grad}
    # Adam over the minibatches, drawn with replacement by the counter-based hash
    n, batch, steps = case["n"], case["batch"], -(-case["n"] // case["batch"])
    m, v, total = torch.zeros_like(p), torch.zeros_like(p), 0.0
    for t in range(steps * case["epochs"]):
        with np.errstate(over="ignore"):
            at = _splitmix(_splitmix(17 + t) + np.arange(batch, dtype=np.uint64)) % np.uint64(n)
        at = torch.from_numpy(at.astype(np.int64)).cuda()
        loss, g = _loss_grad(p, F[at], P[at], T[at])
        total += loss / steps if t < steps else 0.0
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        p = p - 1e-3 * (m / (1 - 0.9 ** (t + 1))) / ((v / (1 - 0.999 ** (t + 1))).sqrt() + 1e-8)
    return {"loss": np.array([total]), "params": p}
