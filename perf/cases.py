"""What a user of this library has it do, as measurable cases.

A case names a workload (the data's recipe), its sizes, the floating type and the call:

* ``train``  -- ``qp_forward`` then ``qp_backward``: the pair behind one training step through
  the layer; returns the solution, the statuses and the six gradients.
* ``infer``  -- ``qp_forward`` alone.
* ``layer``  -- the ``QPFunction`` autograd layer, forward and backward.
* ``module`` -- a training step of ``LearnedEqualityQP`` (forward, MSE, backward).
* ``packed`` -- ``PackedBatch.forward`` / ``.backward`` on a batch of uneven sizes.

Iteration counts and the final residual norms are diagnostics at rounding level and are not
among the outputs; the status codes are.

``exact`` solves the same problems in 64 bits with torch alone: an interior point method finds
the active set, and one KKT solve on that set gives the solution and the adjoint.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1703_00443_gb300 import QPFunction, inputs, qp_backward, qp_forward
from paper_1703_00443_gb300.layers import LearnedEqualityQP
from paper_1703_00443_gb300.packed import PackedBatch

DEV = "cuda"


def _fixed(name, call, data, dtype, batch, n, nineq, neq):
    c = {"call": call, "data": data, "dtype": dtype, "batch": batch, "n": n, "nineq": nineq,
         "neq": neq}
    return dict(c, name=name) if name else c


def _packed(name, data, count, sizes_seed):
    c = {"call": "packed", "data": data, "dtype": "float32", "count": count,
         "sizes_seed": sizes_seed}
    return dict(c, name=name) if name else c


def listed():
    f32, f64 = "float32", "float64"
    return [
        # The smallest layers: ten variables, where launches and dependent steps are the cost.
        _fixed("n10_b128", "train", "random", f32, 128, 10, 10, 5),
        # A small layer at a mid batch.
        _fixed("n50_b64", "train", "random", f32, 64, 50, 50, 25),
        # The headline: one training step through a 100-variable layer, batch 128.
        _fixed("n100_b128", "train", "random", f32, 128, 100, 100, 50),
        # One QP at a time: a control loop or a sequential sampler.
        _fixed("n100_b1", "train", "random", f32, 1, 100, 100, 50),
        # Inference only, odd sizes and batch, inequalities outnumbering the variables.
        _fixed("n77_b100_infer", "infer", "random", f32, 100, 77, 93, 13),
        # One large QP.
        _fixed("n500_b1", "train", "random", f32, 1, 500, 500, 250),
        # A batch of large QPs: the largest fixed-size work.
        _fixed("n500_b128", "train", "random", f32, 128, 500, 500, 250),
        # Training a Sudoku-shaped layer (z >= 0, learned dense equalities), batch 512.
        _fixed("onehot_b512", "module", "onehot", f32, 512, 64, 64, 40),
        # Total-variation denoising of 64 signals of 24 samples: Q only semidefinite.
        _fixed("tv24_b64", "layer", "tv", f32, 64, 47, 46, 0),
        # Double precision, the plain method: eight QPs of ten variables.
        _fixed("fp64_n10_b8", "train", "random", f64, 8, 10, 20, 0),
        # A batch of uneven sizes, n in 8..256, in one packed call each way.
        _packed("uneven_512", "uneven", 512, 0),
        # A served batch: requests with n log-uniform in 16..512.
        _packed("served_256", "serve", 256, 0),
    ]


def draw(rng):
    def logint(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    most = max(work(c)["flops"] for c in listed())
    kind = rng.choices(("train", "infer", "layer", "fp64", "module", "tv", "uneven", "serve"),
                       (6, 3, 2, 2, 2, 1, 2, 2))[0]
    if kind in ("uneven", "serve"):
        count = logint(32, 512) if kind == "uneven" else logint(16, 256)
        return _packed(None, kind, count, rng.randrange(1, 1000))
    if kind == "module":
        n = rng.randrange(16, 97)
        return _fixed(None, "module", "onehot", "float32", logint(16, 512), n, n,
                      max(1, int(n * rng.uniform(0.2, 0.65))))
    if kind == "tv":
        s = rng.randrange(8, 49)
        return _fixed(None, "layer", "tv", "float32", logint(4, 128), 2 * s - 1, 2 * (s - 1), 0)
    if kind == "fp64":
        n = logint(5, 64)
        return _fixed(None, "train", "random", "float64", logint(1, 128), n,
                      max(1, int(n * rng.uniform(0.5, 2.0))), int(n * rng.uniform(0.0, 0.5)))
    n = logint(8, 500)
    c = _fixed(None, kind, "random", "float32", logint(1, 512 if n <= 100 else 128), n,
               max(1, int(n * rng.uniform(0.5, 1.5))), int(n * rng.uniform(0.0, 0.5)))
    while work(c)["flops"] > most and c["batch"] > 1:
        c["batch"] //= 2
    return c


# ---------------------------------------------------------------- problem data
def _sizes(case):
    if case["call"] != "packed":
        return [(case["n"], case["nineq"], case["neq"])] * case["batch"]
    if case["data"] == "uneven":
        return inputs.uneven_sizes(case["count"], seed=case["sizes_seed"])
    return inputs.serve_sizes(case["count"], seed=case["sizes_seed"])


def _random(gen, B, n, p, m, dtype):
    """The §4.1 recipe: Q = L Lᵀ + 1e-3·I, normal G and A, strictly feasible."""
    def nrm(*s):
        return torch.randn(s, generator=gen, device=DEV, dtype=torch.float64)
    L = nrm(B, n, n) / math.sqrt(n)
    Q = L @ L.transpose(1, 2) + 1e-3 * torch.eye(n, device=DEV, dtype=torch.float64)
    Q = (0.5 * (Q + Q.transpose(1, 2))).to(dtype)
    q, G, A, z0 = (x.to(dtype) for x in (nrm(B, n), nrm(B, p, n), nrm(B, m, n), nrm(B, n)))
    s0 = 0.5 + torch.rand((B, p), generator=gen, device=DEV, dtype=torch.float64)
    zd = z0.double().unsqueeze(2)
    h = ((G.double() @ zd).squeeze(2) + s0).to(dtype)
    b = (A.double() @ zd).squeeze(2).to(dtype)
    return [x.contiguous() for x in (Q, q, G, h, A, b)]


def _tv(gen, B, n, dtype):
    """½‖y − z‖² + w·1ᵀt, |Dz| ≤ t, on noisy piecewise-constant signals (§4.2)."""
    s = (n + 1) // 2
    k = s - 1
    t = torch.arange(s, device=DEV).unsqueeze(0)
    cuts = torch.rand((B, 2), generator=gen, device=DEV, dtype=torch.float64).sort(1).values * s
    lev = 2 * torch.rand((B, 3), generator=gen, device=DEV, dtype=torch.float64) - 1
    idx = (t >= cuts[:, :1]).long() + (t >= cuts[:, 1:]).long()
    y = lev.gather(1, idx) + 0.2 * torch.randn((B, s), generator=gen, device=DEV,
                                               dtype=torch.float64)
    Q = torch.zeros((B, n, n), device=DEV, dtype=dtype)
    Q[:, torch.arange(s), torch.arange(s)] = 1
    q = torch.cat([-y, torch.full((B, k), 0.3, device=DEV, dtype=torch.float64)], 1).to(dtype)
    D = torch.diff(torch.eye(s, device=DEV, dtype=torch.float64), dim=0)
    I = torch.eye(k, device=DEV, dtype=torch.float64)
    G = torch.cat([torch.cat([D, -I], 1), torch.cat([-D, -I], 1)], 0).to(dtype)
    return [Q, q, G.expand(B, 2 * k, n).contiguous(), torch.zeros((B, 2 * k), device=DEV, dtype=dtype)]


def _data(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    dtype = getattr(torch, case["dtype"])
    if case["call"] == "packed":
        inst, g = [], []
        for n, p, m in _sizes(case):
            inst.append([x[0] for x in _random(gen, 1, n, p, m, dtype)])
            g.append(torch.randn(n, generator=gen, device=DEV, dtype=dtype))
        return inst, g
    B, n, p, m = (case[k] for k in ("batch", "n", "nineq", "neq"))
    if case["data"] == "onehot":
        A = torch.randn((m, n), generator=gen, device=DEV, dtype=dtype)
        u = torch.rand(n, generator=gen, device=DEV, dtype=dtype)
        x = torch.randn((B, n), generator=gen, device=DEV, dtype=dtype)
        target = torch.rand((B, n), generator=gen, device=DEV, dtype=dtype)
        return A, u, x, target
    T = _tv(gen, B, n, dtype) if case["data"] == "tv" else _random(gen, B, n, p, m, dtype)
    return T, torch.randn((B, n), generator=gen, device=DEV, dtype=dtype)


def prepare(case, seed):
    if case["call"] == "packed":
        inst, g = _data(case, seed)
        pb = PackedBatch(_sizes(case), device=DEV)
        return {"call": "packed", "pb": pb, "T": pb.pack(inst), "g": pb.pack_vec(g, "q")}
    if case["call"] == "module":
        A, u, x, target = _data(case, seed)
        net = LearnedEqualityQP(case["n"], case["neq"], A, u)
        return {"call": "module", "net": net, "x": x.requires_grad_(), "target": target}
    T, g = _data(case, seed)
    if case["call"] == "layer":
        T = [t.requires_grad_() for t in T]
    return {"call": case["call"], "T": T, "g": g}


def run(state):
    call = state["call"]
    if call == "packed":
        pb, T = state["pb"], state["T"]
        f = pb.forward(*T)
        grads = pb.backward(T[0], T[2], T[4], state["g"])
        return {"z": f.z, "lam": f.lam, "nu": f.nu, "status": f.status, "grads": list(grads)}
    if call == "module":
        net, x = state["net"], state["x"]
        z = net(x)
        loss = torch.nn.functional.mse_loss(z, state["target"])
        dA, dx = torch.autograd.grad(loss, (net.A, x))
        return {"z": z.detach(), "loss": loss.detach(), "grads": [dA, dx]}
    if call == "layer":
        z, lam, nu, status = QPFunction.apply(*state["T"], *([None] * (6 - len(state["T"]))))
        grads = torch.autograd.grad(z, state["T"], state["g"])
        return {"z": z.detach(), "lam": lam.detach(), "nu": nu.detach(), "status": status,
                "grads": list(grads)}
    f = qp_forward(*state["T"])
    out = {"z": f.z, "lam": f.lam, "nu": f.nu, "status": f.status}
    if call == "train":
        out["grads"] = list(qp_backward(f, state["g"]))
    return out


def work(case):
    """Bytes: each input read once, each output written once.  FLOPs: one elimination of the
    constant KKT blocks, twelve interior point steps (a Cholesky factorisation of the
    inequalities' Schur complement, two solves and a residual each) and the adjoint solve."""
    esz = 8 if case["dtype"] == "float64" else 4
    nbytes = flops = 0.0
    for n, p, m in _sizes(case):
        vec = n + p + m
        data = n * n + (p + m) * n
        setup = n ** 3 / 3 + n * n * (p + m) + m * m * n / 2 + m ** 3 / 3 + m * p * n + \
            p * n * (n + p + m) / 2
        step = p ** 3 / 6 + 2 * (p * p + 2 * n * (p + m) + n * n)
        flops += 2 * (setup + 12 * step + (0 if case["call"] == "infer" else step - p ** 3 / 6))
        back = 0 if case["call"] == "infer" else (n + data + vec) * esz
        nbytes += (data + 2 * vec) * esz + 4 + back
    if case["call"] == "module":   # the matrices are shared by the batch, and so are their gradients
        n, m, B = case["n"], case["neq"], case["batch"]
        nbytes = 4.0 * (2 * n * n + 2 * m * n + n + 4 * B * n)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- 64-bit values
def _kkt(Q, G, A, act, pad):
    """[Q Gᵀ Aᵀ; act·G I−act 0; A 0 −pad]: the KKT system with the active set's rows."""
    B, n, p, m = Q.shape[0], Q.shape[1], G.shape[1], A.shape[1]
    K = Q.new_zeros((B, n + p + m, n + p + m))
    K[:, :n, :n] = Q
    K[:, :n, n:n + p] = G.transpose(1, 2)
    K[:, :n, n + p:] = A.transpose(1, 2)
    K[:, n:n + p, :n] = G * act.unsqueeze(2)
    K[:, n:n + p, n:n + p] = torch.diag_embed(1.0 - act)
    K[:, n + p:, :n] = A
    K[:, n + p:, n + p:] = torch.diag_embed(-pad)
    return K


def _solve(Q, q, G, h, A, b, pad):
    """z*, λ*, ν* and the KKT matrix on the active set (float64).  pad: 1 on the padding rows
    of A, 0 elsewhere."""
    n, p = Q.shape[1], G.shape[1]
    Gt, At = G.transpose(1, 2), A.transpose(1, 2)

    def mv(M, x):
        return (M @ x.unsqueeze(2)).squeeze(2)

    def factor(w):   # block elimination of [H Aᵀ; A −pad], H = Q + Gᵀ diag(w) G
        C, _ = torch.linalg.cholesky_ex(Q + Gt @ (w.unsqueeze(2) * G))
        W = torch.cholesky_solve(At, C)
        return C, W, torch.linalg.cholesky_ex(A @ W + torch.diag_embed(pad))[0]

    def solve(f, r1, r2):
        C, W, CA = f
        y = torch.cholesky_solve(r1.unsqueeze(2), C).squeeze(2)
        dn = torch.cholesky_solve((mv(A, y) - r2).unsqueeze(2), CA).squeeze(2)
        return y - mv(W, dn), dn

    def direction(f, s, lam, rz, rl, rn, rc):
        # GΔz + Δs = −rl, λΔs + sΔλ = −rc
        dz, dn = solve(f, -rz - mv(Gt, (lam * rl - rc) / s), -rn)
        ds = -rl - mv(G, dz)
        return dz, ds, (-rc - lam * ds) / s, dn

    def longest(v, dv):
        return torch.where(dv < 0, -v / dv, torch.inf).amin(1, keepdim=True)

    z, nu = solve(factor(torch.ones_like(h)), mv(Gt, h) - q, b)
    s = h - mv(G, z)
    s = s + (1.0 - s.amin(1, keepdim=True)).clamp_min(0)
    lam, live = torch.ones_like(s), torch.ones_like(s[:, :1], dtype=torch.bool)
    for _ in range(60):
        rz = mv(Q, z) + q + mv(Gt, lam) + mv(At, nu)
        rl, rn, mu = mv(G, z) + s - h, mv(A, z) - b - pad * nu, (s * lam).mean(1, keepdim=True)
        far = torch.stack([rz.abs().amax(1), rl.abs().amax(1)]).amax(0).unsqueeze(1)
        go = (mu > 1e-10) | (far > 1e-7)
        if not bool((go & live).any()):
            break
        f = factor(lam / s)
        _, ds, dl, _ = direction(f, s, lam, rz, rl, rn, s * lam)
        a = torch.minimum(longest(s, ds), longest(lam, dl)).clamp_max(1.0)
        sig = (((s + a * ds) * (lam + a * dl)).mean(1, keepdim=True) / mu) ** 3
        dz, ds, dl, dn = direction(f, s, lam, rz, rl, rn, s * lam + ds * dl - sig * mu)
        a = (0.99 * torch.minimum(longest(s, ds), longest(lam, dl))).clamp_max(1.0)
        # an instance stops at its last iterate when its elimination breaks down
        live = live & go & torch.isfinite(torch.cat([dz, ds, dl, dn], 1)).all(1, keepdim=True)
        z, s, lam, nu = (torch.where(live, v + a * dv, v)
                         for v, dv in ((z, dz), (s, ds), (lam, dl), (nu, dn)))
    # The active set, corrected until every multiplier and every slack is non-negative: a pair
    # whose larger member is below √μ may sit on the wrong side of the interior iterate.
    act = (lam > s).to(Q.dtype)
    for _ in range(12):
        K = _kkt(Q, G, A, act, pad)
        rhs = torch.cat([-q, act * h, b], 1).unsqueeze(2)
        lu = torch.linalg.lu_factor_ex(K)[:2]
        x = torch.linalg.lu_solve(*lu, rhs)
        x = (x + torch.linalg.lu_solve(*lu, rhs - K @ x)).squeeze(2)
        wrong = torch.where(act > 0, x[:, n:n + p] < 0,
                            h - mv(G, x[:, :n]) < -1e-12 * (1 + h.abs()))
        if not bool(wrong.any()):
            break
        act = torch.where(wrong, 1 - act, act)
    return x[:, :n], x[:, n:n + p], x[:, n + p:], K, lu


def _values(Q, q, G, h, A, b, pad, g):
    """(z, λ, ν, dQ, dq, dG, dh, dA, db) in float64; g: ∂ℓ/∂z*, or a function of z*, or None."""
    n, p = Q.shape[1], G.shape[1]
    z, lam, nu, K, lu = _solve(Q, q, G, h, A, b, pad)
    if g is None:
        return z, lam, nu
    if callable(g):
        g = g(z)
    rhs = torch.cat([-g, torch.zeros_like(h), torch.zeros_like(b)], 1).unsqueeze(2)
    d = torch.linalg.lu_solve(*lu, rhs)
    d = (d + torch.linalg.lu_solve(*lu, rhs - K @ d)).squeeze(2)
    dz, dl, dn = d[:, :n], d[:, n:n + p], d[:, n + p:]

    def outer(x, y):
        return x.unsqueeze(2) * y.unsqueeze(1)
    return (z, lam, nu, 0.5 * (outer(dz, z) + outer(z, dz)), dz, outer(dl, z) + outer(lam, dz),
            -dl, outer(dn, z) + outer(nu, dz), -dn)


def _padded(inst, g):
    """Instances of one chunk, padded to its largest sizes: dummy variables with Q = 1,
    inequalities 0 ≤ 1 and multipliers fixed at 0."""
    B = len(inst)
    n, p, m = (max(t[k].shape[0] for t in inst) for k in (1, 3, 5))
    def z(*s):
        return torch.zeros((B, *s), device=DEV, dtype=torch.float64)
    Q, q, G, h, A, b, pad, gg = z(n, n), z(n), z(p, n), z(p) + 1, z(m, n), z(m), z(m) + 1, z(n)
    Q += torch.eye(n, device=DEV, dtype=torch.float64)
    for i, (t, gi) in enumerate(zip(inst, g)):
        ni, pi, mi = t[1].shape[0], t[3].shape[0], t[5].shape[0]
        Q[i, :ni, :ni], q[i, :ni], G[i, :pi, :ni], h[i, :pi] = t[0], t[1], t[2], t[3]
        A[i, :mi, :ni], b[i, :mi], pad[i, :mi], gg[i, :ni] = t[4], t[5], 0, gi
    return Q, q, G, h, A, b, pad, gg


def exact(case, seed):
    if case["call"] == "packed":
        inst, g = _data(case, seed)
        sizes = np.array(_sizes(case))
        vals = [None] * len(inst)
        for ch in np.array_split(np.argsort(sizes.sum(1), kind="stable"),
                                 max(1, len(inst) // 32)):
            v = _values(*_padded([inst[i] for i in ch], [g[i] for i in ch]))
            for k, i in enumerate(ch):
                n, p, m = sizes[i]
                cut = ((n,), (p,), (m,), (n, n), (n,), (p, n), (p,), (m, n), (m,))
                vals[i] = [x[k][tuple(slice(0, int(e)) for e in c)] for x, c in zip(v, cut)]

        def flat(j):   # each instance's values start at a multiple of four elements
            total = sum(-(-v[j].numel() // 4) * 4 for v in vals)
            out, o = torch.zeros(max(1, total), device=DEV, dtype=torch.float64), 0
            for v in vals:
                out[o:o + v[j].numel()] = v[j].reshape(-1)
                o += -(-v[j].numel() // 4) * 4
            return out
        return {"z": flat(0), "lam": flat(1), "nu": flat(2), "status": None,
                "grads": [flat(j) for j in range(3, 9)]}
    if case["call"] == "module":
        A, u, x, target = (t.double() for t in _data(case, seed))
        B, n, m = case["batch"], case["n"], case["neq"]
        I = torch.eye(n, device=DEV, dtype=torch.float64)
        # the layer holds 0.1·I and b = A u in its own type
        Q = torch.tensor(0.1, dtype=getattr(torch, case["dtype"])).double().to(DEV) * I
        z, _, _, _, dq, _, _, dA, db = _values(
            Q.expand(B, n, n), x, (-I).expand(B, n, n), torch.zeros_like(x), A.expand(B, m, n),
            (A @ u).expand(B, m), torch.zeros((B, m), device=DEV, dtype=torch.float64),
            lambda zz: 2 * (zz - target) / zz.numel())
        dA = dA.sum(0) + torch.outer(db.sum(0), u)
        return {"z": z, "loss": ((z - target) ** 2).mean(), "grads": [dA, dq]}
    T, g = _data(case, seed)
    T, g, given = [t.double() for t in T], g.double(), len(T)
    if given == 4:
        T += [torch.zeros((T[0].shape[0], 0, T[0].shape[1]), device=DEV, dtype=torch.float64),
              torch.zeros((T[0].shape[0], 0), device=DEV, dtype=torch.float64)]
    v = _values(*T, torch.zeros_like(T[5]), None if case["call"] == "infer" else g)
    out = {"z": v[0], "lam": v[1], "nu": v[2], "status": None}
    if case["call"] != "infer":
        out["grads"] = list(v[3:3 + given])
    return out
