"""What a user of this library has it do, as cases that can be timed.

A case is a plain dict.  ``listed()`` gives the fixed ones, ``draw(rng)`` one
more of the same ranges, ``prepare(case, seed)`` the state a program holds
before the call (inputs from the seed alone), ``run(state)`` one pass through
the public entry points, ``work(case)`` the bytes and floating-point
operations the path cannot do without, ``exact(case, seed)`` the outputs as
plain numpy / torch gives them in 64 bits without this package's library.

Kinds:
  todm    host gate list to density matrix and <O> (Stab.apply_circuit, expect,
          density_matrix), the paper's toDM() call
  step    new angles in device memory, then the n generators and <O>
  expect  new angles in device memory, then <O>
  grad    new angles in device memory, then <O> and the adjoint gradient (a
          training step)
  batch   many uneven circuits in one launch: the parameter-shift copies of
          one circuit, further <O> items, and generator items
  serve   a burst of uneven <O> and gradient requests through the server
  sparse  <O> and one generator of a wide circuit held as term lists
"""
import math

import numpy as np
import torch

from paper_2502_10685_gb300 import stab, workloads as W

MAX_UNITS = 2.2e8   # gates x 4^n of the largest dense single-circuit case drawn


def listed():
    return [
        # the smallest call: a short 2-qubit circuit from host gates to the host density matrix
        {"name": "todm-n2-100", "kind": "todm", "n": 2, "m": 100, "circuit": "layered",
         "obs": "chain"},
        # the paper's small layered ansatz: 4 generators and <O> at new angles
        {"name": "step-n4-2000", "kind": "step", "n": 4, "m": 2000, "circuit": "layered",
         "obs": "z0"},
        # the paper's headline circuit size (60,200 gates on 4 qubits)
        {"name": "step-n4-60200", "kind": "step", "n": 4, "m": 60200, "circuit": "layered",
         "obs": "z0z1"},
        # vectors too large for one SM: 9 generators streamed through memory
        {"name": "step-n9-1001", "kind": "step", "n": 9, "m": 1001, "circuit": "layered",
         "obs": "chain"},
        # the largest register: one 4^12 observable through a shallow circuit
        {"name": "expect-n12-400", "kind": "expect", "n": 12, "m": 400, "circuit": "layered",
         "obs": "chain"},
        # training steps: small register, the size on the edge of residency, the
        # 10,000-gate n = 8 differentiation workload, and a large register
        {"name": "grad-n4-4000", "kind": "grad", "n": 4, "m": 4000, "circuit": "layered",
         "obs": "chain"},
        {"name": "grad-n6-2003", "kind": "grad", "n": 6, "m": 2003, "circuit": "layered",
         "obs": "chain"},
        {"name": "grad-n8-10000", "kind": "grad", "n": 8, "m": 10000, "circuit": "layered",
         "obs": "chain"},
        {"name": "grad-n10-600", "kind": "grad", "n": 10, "m": 600, "circuit": "layered",
         "obs": "chain"},
        # parameter-shift copies and uneven circuits in one persistent launch
        {"name": "batch-600", "kind": "batch", "n": 6, "m": 400, "variants": 500, "items": 76,
         "gens": 24, "deep": 8000},
        # a burst of requests on the serving engine
        {"name": "serve-48", "kind": "serve", "n": 8, "m": 6000, "requests": 48},
        # 32 qubits as a term list: Clifford gates with few rotations
        {"name": "sparse-n32-20000", "kind": "sparse", "n": 32, "m": 20000, "rot": 28},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["todm", "step", "step", "expect", "expect", "grad", "grad", "grad",
                       "batch", "serve", "sparse"])
    if kind == "sparse":
        return {"kind": kind, "n": rng.randint(13, 32), "m": _log_int(rng, 300, 20000),
                "rot": rng.randint(8, 28)}
    if kind == "serve":
        return {"kind": kind, "n": rng.randint(5, 8), "m": _log_int(rng, 300, 6000),
                "requests": rng.randint(6, 48)}
    if kind == "batch":
        return {"kind": kind, "n": rng.randint(2, 6), "m": _log_int(rng, 60, 400),
                "variants": _log_int(rng, 16, 500), "items": rng.randint(4, 76),
                "gens": rng.randint(1, 24), "deep": _log_int(rng, 300, 8000)}
    n = {"todm": rng.randint(1, 6), "step": rng.randint(1, 10), "expect": rng.randint(2, 12),
         "grad": rng.randint(2, 11)}[kind]
    cost = {"todm": 1, "step": n, "expect": 1, "grad": 3}[kind] * 4 ** n
    top = int(min(60200, max(150, MAX_UNITS / cost)))
    m = _log_int(rng, 100, top)
    return {"kind": kind, "n": n, "m": m,
            "circuit": rng.choice(["layered", "layered", "paper", "random", "shared"]),
            "obs": rng.choice(["chain", "z0", "terms"])}


# ---------------------------------------------------------------- inputs

def _angles(c, seed):
    """The circuit at the seed's angles.  Which gate sits where follows from
    the case (outputs keep their shapes); the angles are the seed's."""
    th = np.random.default_rng(seed).uniform(0.0, 2.0 * math.pi, c.n_params)
    return c.with_thetas(th)


def _circuit(case, seed):
    n, m, form = case["n"], case["m"], case.get("circuit", "layered")
    key = 1000 * m + n
    if form == "layered":
        c = W.layered_ansatz(n, m, key)
    elif form == "paper":
        # W_chain + ZXZ blocks, a few repeats per layer, cut to about m gates
        reps = 1 + key % 7
        per = (n if n > 1 else 0) + 3 * n * reps
        c = W.paper_shaped_ansatz(n, max(1, m // per), reps, key)
    else:
        c = W.random_circuit(n, m, key, shared_params=(max(1, m // 9) if form == "shared" else 0))
    return _angles(c, seed)


def _sparse_circuit(case, seed):
    n, m, rot = case["n"], case["m"], case["rot"]
    return _angles(W.clifford_plus_rotations(n, m, rot, 1000 * m + 100 * n + rot), seed)


def _observable(case, seed):
    n, form = case["n"], case.get("obs", "chain")
    if form == "z0":
        return W.obs_z(n, 0)
    if form == "z0z1":
        return W.obs_zz(n, 0, 1)
    if form == "terms":
        return W.random_observable(n, 12, seed + 3) + W.obs_chain(n)
    return W.obs_chain(n)


def _batch_items(case, seed):
    """Parameter-shift copies of one circuit, uneven <O> items, generator items."""
    n, key = case["n"], 1000 * case["m"] + case["n"]
    rng = np.random.default_rng(key)
    base = _angles(W.layered_ansatz(n, case["m"], key), seed)
    items = [W.BatchItem(v, "expect", W.obs_chain(n))
             for v in W.psr_variants(base)[:case["variants"]]]
    for k in range(case["items"] + case["gens"]):
        gens = k >= case["items"]
        nn = int(rng.integers(2, 7 if gens else 9))
        depth = int(round(math.exp(rng.uniform(math.log(100), math.log(case["deep"])))))
        c = _angles(W.layered_ansatz(nn, depth, key + 100 + k), seed + 100 + k)
        items.append(W.BatchItem(c, "generators") if gens
                     else W.BatchItem(c, "expect", W.obs_chain(nn)))
    return items


def _requests(case, seed):
    # half of them <O>, half gradients, whatever the seed
    trace = W.serving_trace(case["requests"], case["m"], n_range=(4, case["n"]),
                            depth_range=(100, case["m"]))
    return [(_angles(r.circuit, seed + k), "grad" if k % 2 else "expect", r.observable)
            for k, r in enumerate(trace)]


# ---------------------------------------------------------------- state and pass

def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind}
    if kind == "batch":
        items = _batch_items(case, seed)
        st["batch"] = stab.Batch(items)
        st["gens"] = [k for k, it in enumerate(items) if it.kind == "generators"]
        return st
    if kind == "serve":
        st["server"] = stab.Server(policy="shortest")
        st["requests"] = _requests(case, seed)
        return st
    if kind == "sparse":
        c = _sparse_circuit(case, seed)
        s = stab.Sparse(case["n"])
        s.load_circuit(c.gates, c.thetas)
        st.update(s=s, obs=W.obs_chain(case["n"]))
        return st
    c, obs = _circuit(case, seed), _observable(case, seed)
    s = stab.Stab(case["n"])
    st.update(s=s, c=c, obs=obs)
    if kind == "todm":
        return st
    # a program that trains or scans angles: the circuit is loaded once, the
    # angles live on the device
    s.load_circuit(c.gates, np.zeros(c.n_params))
    s.set_observable(obs)
    st["thetas"] = torch.tensor(c.thetas, dtype=torch.float64, device="cuda")
    st["e"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    if kind == "step":
        st["out"] = torch.zeros(c.n, 4 ** c.n, dtype=torch.float64, device="cuda")
    if kind == "grad":
        st["out"] = torch.zeros(max(1, c.n_params), dtype=torch.float64, device="cuda")
    return st


def run(st):
    kind = st["kind"]
    if kind == "batch":
        b = st["batch"]
        b.run()
        return {"expect": b.expectations(), "gens": [b.generators(k) for k in st["gens"]]}
    if kind == "serve":
        srv = st["server"]
        ids = [srv.submit(c, kind, obs) for c, kind, obs in st["requests"]]
        res = [srv.wait(i) for i in ids]
        return {"status": np.array([r["status"] for r in res]),
                "expect": np.array([r["expect"] for r in res]),
                "grads": np.concatenate([r["grads"] for r, q in zip(res, st["requests"])
                                         if q[1] == "grad"] or [np.zeros(1)])}
    s = st["s"]
    if kind == "sparse":
        value, info = s.expect(st["obs"])
        terms, _ = s.generator(0)
        return {"expect": value, "order": info["order_final"], "coeff": terms["coeff"],
                "x": terms["x"].astype(np.int64), "z": terms["z"].astype(np.int64)}
    if kind == "todm":
        c = st["c"]
        s.apply_circuit(c.gates, c.thetas)
        return {"expect": s.expect(st["obs"]), "rho": s.density_matrix()}
    s.set_params(st["thetas"])
    if kind == "step":
        s.run_generators()
        s.expect_async(st["e"])
        s.generators(out=st["out"])
        return {"expect": st["e"], "gens": st["out"]}
    if kind == "expect":
        s.expect_async(st["e"])
        return {"expect": st["e"]}
    s.grad_async(st["e"], st["out"])
    return {"expect": st["e"], "grads": st["out"]}


# ---------------------------------------------------------------- work

def _rot_share(case):
    # share of the gates that are rotations, by construction of the circuits
    form, n = case.get("circuit", "layered"), case["n"]
    if form in ("random", "shared"):
        return 6.0 / 14.0 if n > 1 else 6.0 / 12.0
    if form == "paper":
        return 0.9
    return 0.675 if n > 1 else 0.9


def _grad_flops(rot, n):
    # lambda and rho through every rotation (1.5 x 4^n each), and its inner
    # product over the rotation's pairs (4 operations a pair, 4^n / 4 pairs)
    return rot * 4.0 ** n * (2 * 1.5 + 1.0)


def work(case):
    kind, n, m = case["kind"], case["n"], case["m"]
    E = 4.0 ** n
    if kind == "sparse":
        # the chain's terms and one generator, half of them doubled by each
        # rotation: reads and writes of the last lists (16-byte terms), the
        # rotations' products
        order = 2 * n * 1.5 ** case["rot"]
        return {"bytes": 8.0 * m + 3 * 32.0 * order, "flops": 6.0 * order}
    if kind == "batch":
        mean_depth = (case["deep"] - 100.0) / math.log(case["deep"] / 100.0)
        flops = case["variants"] * m * 0.675 * 1.5 * E
        flops += case["items"] * mean_depth * 0.675 * 1.5 * sum(4.0 ** k for k in range(2, 9)) / 7
        flops += case["gens"] * mean_depth * 0.675 * 1.5 * sum(k * 4.0 ** k
                                                              for k in range(2, 7)) / 5
        gates = case["variants"] * m + (case["items"] + case["gens"]) * mean_depth
        return {"bytes": 8.0 * gates, "flops": flops}
    if kind == "serve":
        mean_depth = (m - 100.0) / math.log(m / 100.0)
        per = sum(0.5 * 0.675 * mean_depth * 1.5 * 4.0 ** k
                  + 0.5 * _grad_flops(0.675 * mean_depth, k) for k in range(4, n + 1)) / (n - 3)
        return {"bytes": case["requests"] * mean_depth * 16.0, "flops": case["requests"] * per}
    rot = _rot_share(case) * m
    if kind == "todm":
        return {"bytes": 8.0 * m + 8.0 * rot + 16.0 * E, "flops": rot * 1.5 * E}
    if kind == "step":
        return {"bytes": 8.0 * rot + 8.0 * n * E, "flops": (n + 1) * rot * 1.5 * E}
    if kind == "expect":
        return {"bytes": 8.0 * rot, "flops": rot * 1.5 * E}
    return {"bytes": 16.0 * rot, "flops": _grad_flops(rot, n)}


# ---------------------------------------------------------------- 64-bit values
#
# Plain state-vector arithmetic in complex128 (bit q of an index is qubit q),
# R_s(theta) = exp(-i theta s / 2).

_SQ = 1.0 / math.sqrt(2.0)
_FIXED = {0: [[_SQ, _SQ], [_SQ, -_SQ]], 1: [[1, 0], [0, 1j]], 2: [[1, 0], [0, -1j]],
          3: [[0, 1], [1, 0]], 4: [[0, -1j], [1j, 0]], 5: [[1, 0], [0, -1]]}
_FIXED = {k: np.array(v, dtype=np.complex128) for k, v in _FIXED.items()}
_SIGMA = {8: 3, 9: 4, 10: 5}


def _matrix(op, theta):
    if op < 6:
        return _FIXED[op]
    c, s = math.cos(theta / 2), math.sin(theta / 2)
    if op == 8:
        return np.array([[c, -1j * s], [-1j * s, c]])
    if op == 9:
        return np.array([[c, -s], [s, c]], dtype=np.complex128)
    return np.array([[complex(c, -s), 0], [0, complex(c, s)]])


def _apply1(v, q, M):
    """A 2 x 2 matrix on qubit q of the first axis of v (2^n, columns)."""
    w = v.reshape(v.shape[0] >> (q + 1), 2, 1 << q, -1)
    a, b = w[:, 0], w[:, 1]
    out = np.empty_like(w)
    out[:, 0] = M[0, 0] * a + M[0, 1] * b
    out[:, 1] = M[1, 0] * a + M[1, 1] * b
    return out.reshape(v.shape)


def _apply2(v, op, a, b):
    idx = np.arange(v.shape[0])
    if op == 6:
        return v[idx ^ (((idx >> a) & 1) << b)]
    return v * (1.0 - 2.0 * ((idx >> a) & (idx >> b) & 1)).reshape(-1, *[1] * (v.ndim - 1))


def _records(c):
    g = c.gates
    return zip(g["op"].tolist(), g["q0"].tolist(), g["q1"].tolist(), g["param"].tolist())


def _forward(c, v):
    th = c.thetas.tolist()
    for op, a, b, p in _records(c):
        v = _apply2(v, op, a, b) if op in (6, 7) else _apply1(v, a, _matrix(op, th[p] if op > 7
                                                                            else 0.0))
    return v


def _apply_obs(v, obs, n):
    out = np.zeros_like(v)
    idx = np.arange(1 << n)
    for coeff, s in obs:
        x = sum(1 << q for q in range(n) if s[q] in "XY")
        z = sum(1 << q for q in range(n) if s[q] in "ZY")
        par = np.array([bin(i).count("1") & 1 for i in range(1 << n)])
        sign = 1.0 - 2.0 * par[idx & z]
        w = (coeff * 1j ** bin(x & z).count("1")) * sign * v
        out[idx ^ x] += w
    return out


def _zero(n):
    v = np.zeros((1 << n, 1), dtype=np.complex128)
    v[0, 0] = 1.0
    return v


def _expect(c, obs):
    psi = _forward(c, _zero(c.n))[:, 0]
    return float(np.vdot(psi, _apply_obs(psi, obs, c.n)).real)


def _expect_and_grad(c, obs):
    n, th = c.n, c.thetas.tolist()
    psi = _forward(c, _zero(n))
    lam = _apply_obs(psi[:, 0], obs, n).reshape(-1, 1)
    e = float(np.vdot(psi, lam).real)
    grads = np.zeros(max(1, c.n_params))
    pair = np.concatenate([psi, lam], axis=1)
    for op, a, b, p in reversed(list(_records(c))):
        if op in (6, 7):
            pair = _apply2(pair, op, a, b)
            continue
        if op > 7:
            grads[p] += np.vdot(pair[:, 1], _apply1(pair[:, :1], a, _FIXED[_SIGMA[op]])[:, 0]).imag
        pair = _apply1(pair, a, _matrix(op, th[p] if op > 7 else 0.0).conj().T)
    return e, grads


def _pauli_coefficients(A, n):
    """2^-n Tr(P(x, z) A) over all strings at index z | (x << n), real parts."""
    N = 1 << n
    b = np.arange(N)
    rows = A[b[None, :], b[None, :] ^ b[:, None]]        # [x, b] = A[b, b ^ x]
    for q in range(n):
        w = rows.reshape(N, N >> (q + 1), 2, 1 << q)
        rows = np.stack([w[:, :, 0] + w[:, :, 1], w[:, :, 0] - w[:, :, 1]], axis=2).reshape(N, N)
    par = np.array([bin(i).count("1") for i in range(N)])
    phase = np.array([1, 1j, -1, -1j])[par[b[:, None] & b[None, :]] & 3]
    return (phase * rows).real.reshape(-1) / N


def _generators(c):
    n = c.n
    U = _forward(c, np.eye(1 << n, dtype=np.complex128))
    idx = np.arange(1 << n)
    return np.stack([_pauli_coefficients((U * (1.0 - 2.0 * ((idx >> k) & 1))) @ U.conj().T, n)
                     for k in range(n)])


def _sparse_expect(c, obs):
    """The observable as its term list, gate by gate backward (torch, int64 keys)."""
    n, th = c.n, c.thetas.tolist()
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    x = torch.tensor([sum(1 << q for q in range(n) if s[q] in "XY") for _, s in obs], device=dev)
    z = torch.tensor([sum(1 << q for q in range(n) if s[q] in "ZY") for _, s in obs], device=dev)
    co = torch.tensor([float(k) for k, _ in obs], dtype=torch.float64, device=dev)
    for op, a, b, p in reversed(list(_records(c))):
        xa, za = (x >> a) & 1, (z >> a) & 1
        if op in (6, 7):
            xb, zb = (x >> b) & 1, (z >> b) & 1
            if op == 6:
                neg = xa & zb & ((xb ^ za) ^ 1)
                x, z = x ^ (xa << b), z ^ (zb << a)
            else:
                neg = xa & xb & (za ^ zb)
                z = z ^ (xb << a) ^ (xa << b)
        elif op == 0:
            neg = xa & za
            x, z = x ^ ((xa ^ za) << a), z ^ ((xa ^ za) << a)
        elif op == 1:                      # S^dagger P S: X -> -Y, Y -> X
            neg = xa & (za ^ 1)
            z = z ^ (xa << a)
        elif op == 2:
            neg = xa & za
            z = z ^ (xa << a)
        elif op < 6:
            neg = {3: za, 4: xa ^ za, 5: xa}[op]
        else:
            # U^dagger P U for the terms that anticommute with the axis:
            # cos(t) P + i sin(t) / 2 [s, P]
            sx, sz = {8: (1, 0), 9: (1, 1), 10: (0, 1)}[op]
            hit = ((xa & sz) ^ (za & sx)).bool()
            # i s P = sign * Q with Q on letters s * P: +1 for the cyclic pairs
            # (X, Z), (Y, X), (Z, Y) of (s, P), as i X Z = Y and so on
            letter = xa + 2 * za           # 0 I, 1 X, 2 Z, 3 Y
            plus = {8: 2, 9: 1, 10: 3}[op]
            sign = torch.where(letter[hit] == plus, 1.0, -1.0).to(torch.float64)
            c_, s_ = math.cos(th[p]), math.sin(th[p])
            x2, z2, k2 = x[hit] ^ (sx << a), z[hit] ^ (sz << a), co[hit] * sign * s_
            co = torch.where(hit, co * c_, co)
            x, z, co = torch.cat([x, x2]), torch.cat([z, z2]), torch.cat([co, k2])
            key, inv = torch.unique((x << n) | z, return_inverse=True)
            co = torch.zeros(key.numel(), dtype=torch.float64, device=dev).index_add_(0, inv, co)
            x, z = (key >> n) & ((1 << n) - 1), key & ((1 << n) - 1)
            continue
        co = torch.where(neg.bool(), -co, co)
    return float(co[x == 0].sum().item())


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        items = _batch_items(case, seed)
        ex = np.full(len(items), np.nan)
        gens = []
        # the parameter-shift copies differ in their angles only: one sweep over
        # all of them at once, the copies as columns
        nv = len(items) - case["items"] - case["gens"]
        base = items[0].circuit
        th = np.stack([it.circuit.thetas for it in items[:nv]], axis=1)
        v = np.repeat(_zero(base.n), nv, axis=1)
        for op, a, b, p in _records(base):
            if op in (6, 7):
                v = _apply2(v, op, a, b)
            elif op < 6:
                v = _apply1(v, a, _FIXED[op])
            else:
                c_, s_ = np.cos(th[p] / 2), np.sin(th[p] / 2)
                S = _apply1(v, a, _FIXED[_SIGMA[op]])
                v = c_ * v - 1j * s_ * S
        for k in range(nv):
            w = v[:, k]
            ex[k] = np.vdot(w, _apply_obs(w, items[k].observable, base.n)).real
        for k in range(nv, len(items)):
            it = items[k]
            if it.kind == "generators":
                gens.append(_generators(it.circuit))
            else:
                ex[k] = _expect(it.circuit, it.observable)
        return {"expect": ex, "gens": gens}
    if kind == "serve":
        ex, grads = [], []
        for c, what, obs in _requests(case, seed):
            if what == "grad":
                e, g = _expect_and_grad(c, obs)
                grads.append(g[:c.n_params])
            else:
                e = _expect(c, obs)
            ex.append(e)
        return {"status": None, "expect": np.array(ex),
                "grads": np.concatenate(grads or [np.zeros(1)])}
    if kind == "sparse":
        c = _sparse_circuit(case, seed)
        return {"expect": _sparse_expect(c, W.obs_chain(case["n"])), "order": None, "coeff": None,
                "x": None, "z": None}
    c, obs = _circuit(case, seed), _observable(case, seed)
    if kind == "todm":
        psi = _forward(c, _zero(c.n))[:, 0]
        return {"expect": float(np.vdot(psi, _apply_obs(psi, obs, c.n)).real),
                "rho": np.outer(psi, psi.conj())}
    if kind == "grad":
        e, g = _expect_and_grad(c, obs)
        return {"expect": np.array([e]), "grads": g}
    if kind == "expect":
        return {"expect": np.array([_expect(c, obs)])}
    if c.m * 4.0 ** c.n > 2.7e9:
        return None
    return {"expect": np.array([_expect(c, obs)]), "gens": _generators(c)}
