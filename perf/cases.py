"""What is timed: the calls a user of the library makes, over the sizes they make them at.

Most work goes through ``TTN.step`` (one second-order TDVP step with the
populations read back, the loop of every run), in both precisions, from
product states (the start of a circuit, rank-deficient bonds) and from
entangled states (later in a circuit, every bond full).  Around it: reading
the observables, drawing measurement shots, truncating a state, the gradient
of the final fidelity, and the contraction on device buffers.

Inputs are synthetic and made from the seed: product states with random
single-qubit phases, and random isometric trees whose root has a spectrum
falling from 1 to 1e-6 (what a bond of a truncated state looks like).
"""
import math

import numpy as np
import torch

from paper_2210_03763_gb300 import native, workloads as W

DT = 0.01
C6 = 20.0
PREC = {"fp64": native.FP64, "split": native.SPLIT_TF32X3}


# ------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest call: a device-buffer contraction at the 81-wide bonds of level 1
        {"name": "contract_81", "kind": "contract", "M": 81, "N": 81, "K": 81},
        # four atoms: every node fits one block, launches and round trips count
        step("step_2x2_chi16_fp64", 2, 2, 16, "fp64", "product", "layer"),
        # the paper's own bond dimension on its largest lattice: 63 small nodes
        step("step_8x8_chi12_fp64", 8, 8, 12, "fp64", "product", "layer"),
        # GHZ preparation on 16 atoms in FP64, bonds full
        step("step_4x4_chi64_fp64", 4, 4, 64, "fp64", "entangled", "circuit"),
        # the open system (Arnoldi) in split precision
        step("decay_4x4_chi64_split", 4, 4, 64, "split", "entangled", "circuit", gamma=0.2),
        # a lattice that does not fill its tree (35 atoms on 64 leaves), odd bond dimension
        step("step_5x7_chi100_split", 5, 7, 100, "split", "product", "layer"),
        # the benchmark's workload: a parallel CZ layer on 64 atoms
        step("step_8x8_chi128_split", 8, 8, 128, "split", "product", "layer"),
        # the same lattice once the state is entangled: every QR at full rank
        step("step_8x8_chi128_entangled", 8, 8, 128, "split", "entangled", "layer"),
        # what is read between steps: populations of |0> and |r>, norm, energy, GHZ fidelity
        {"name": "observe_8x8_chi128", "kind": "observe", "Lx": 8, "Ly": 8, "chi": 128, "pulses": "layer"},
        # measurement histograms
        {"name": "sample_8x8_chi128_split", "kind": "sample", "Lx": 8, "Ly": 8, "chi": 128, "prec": "split",
         "shots": 64},
        # truncation to a smaller bond dimension (convergence checks)
        {"name": "compress_4x4_chi64_to_16", "kind": "compress", "Lx": 4, "Ly": 4, "chi": 64, "to": 16},
        # pulse optimisation: gradient of the final fidelity over segmented CZ pulses
        {"name": "gradient_3x2_chi27_fp64", "kind": "gradient", "Lx": 3, "Ly": 2, "chi": 27, "prec": "fp64",
         "steps": 3, "quad": 4},
    ]


def step(name, Lx, Ly, chi, prec, start, pulses, gamma=0.0):
    c = {"kind": "step", "Lx": Lx, "Ly": Ly, "chi": chi, "prec": prec, "start": start, "pulses": pulses,
         "gamma": gamma}
    if name:
        c["name"] = name
    return c


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["contract", "observe", "sample", "compress", "gradient"])
    if kind == "contract":
        while True:
            M, N, K = _log(rng, 20, 2000), _log(rng, 16, 400), _log(rng, 16, 1000)
            a, b = max(M, N), min(M, N)
            planes = 2 * (-(-a // 128) * 128 + -(-2 * b // 64) * 64) * (-(-2 * K // 32) * 32) * 4
            if a >= 64 and planes + 4096 < 8 << 20:   # the packed operands the call has room for
                return {"kind": kind, "M": M, "N": N, "K": K}
    if kind == "gradient":
        Lx, Ly, chi = rng.choice([(2, 2, 9), (2, 2, 16), (3, 2, 27), (2, 3, 27)])
        return {"kind": kind, "Lx": Lx, "Ly": Ly, "chi": chi, "prec": "fp64", "steps": rng.randint(1, 5),
                "quad": rng.randint(2, 6)}
    if kind == "step":
        prec = rng.choice(["fp64", "split"])
        start = rng.choice(["product", "entangled"])
        gamma = rng.choice([0.0, 0.0, 0.2])
        if prec == "fp64":
            Lx, Ly = rng.choice([(2, 2), (2, 3), (1, 5), (3, 3), (4, 3), (4, 4), (5, 5), (8, 4), (8, 8)])
            chi = _log(rng, 8, 64 if Lx * Ly <= 16 else 18)
        else:
            Lx, Ly = rng.choice([(4, 3), (4, 4), (5, 4), (5, 5), (8, 4), (6, 6), (7, 7), (8, 8)])
            chi = _log(rng, 32, 128 if Lx * Ly <= 16 else 96)
        pulses = "circuit" if start == "entangled" and (prec == "fp64" or Lx * Ly <= 25) else "layer"
        return step(None, Lx, Ly, chi, prec, start, pulses, gamma)
    Lx, Ly = rng.choice([(3, 3), (4, 4), (5, 4), (8, 4), (6, 6), (8, 8)])
    if kind == "observe":
        return {"kind": kind, "Lx": Lx, "Ly": Ly, "chi": _log(rng, 12, 96), "pulses": "layer"}
    if kind == "sample":
        prec = rng.choice(["split", "fp64"])
        return {"kind": kind, "Lx": Lx, "Ly": Ly, "chi": _log(rng, 12, 128 if prec == "split" else 40), "prec": prec,
                "shots": _log(rng, 4, 256 if prec == "split" else 64)}
    chi = _log(rng, 16, 64)
    return {"kind": kind, "Lx": Lx, "Ly": Ly, "chi": chi, "to": max(2, _log(rng, 4, chi))}


# -------------------------------------------------------------- tree and work
def tree(Lx, Ly, chi):
    """Nodes bottom-up, the root last: (d0, d1, d2, atoms under each child, atoms elsewhere)."""
    N = Lx * Ly
    leaves = 2
    while leaves < N:
        leaves *= 2
    n_at, dim, out = [1 if l < N else 0 for l in range(leaves)], [3] * leaves, []
    while len(n_at) > 1:
        up_n, up_d = [], []
        for i in range(0, len(n_at), 2):
            a = n_at[i] + n_at[i + 1]
            d2 = 1 if len(n_at) == 2 else min(chi, 3 ** a, 3 ** (N - a))
            out.append((dim[i], dim[i + 1], d2, n_at[i], n_at[i + 1], N - a))
            up_n.append(a)
            up_d.append(d2)
        n_at, dim = up_n, up_d
    return out


def _heff(d, n):
    """Flops of one H_eff application to a tensor with legs d and n atoms behind each."""
    s = d[0] * d[1] * d[2]
    f = 8.0 * s * sum(d[u] for u in range(3) if n[u])
    for u, v in ((0, 1), (0, 2), (1, 2)):
        f += 8.0 * s * min(n[u], n[v]) * (d[u] + d[v])
    return f


def _step_work(Lx, Ly, chi):
    """One step with a Krylov space of 4 (about the least that dt = 0.01 needs): every node and link
    evolved twice, four gauge moves and four one-site-operator environments per bond; each tensor and
    environment read once and written once."""
    by = fl = 0.0
    for d0, d1, d2, n0, n1, n2 in tree(Lx, Ly, chi):
        d, s = (d0, d1, d2), d0 * d1 * d2
        fl += 2 * 4 * _heff(d, (n0, n1, n2))
        by += 2 * 16.0 * s
        if d2 > 1 or n2:
            fl += 2 * 4 * _heff((d2, d2, 1), (n0 + n1, n2, 0))
            fl += 4 * 8.0 * s * d2 * 2                                  # QR and absorb, each end, both sweeps
            fl += 2 * 8.0 * s * ((n0 + n1) * (max(d0, d1) + d2))        # n_i towards the parent
            fl += 2 * 8.0 * s * (n1 + n2) * (max(d1, d2) + d0) + 2 * 8.0 * s * (n0 + n2) * (max(d0, d2) + d1)
            by += 2 * 16.0 * d2 * d2 * (n0 + n1 + n2)
    return {"bytes": by, "flops": fl}


def _node_sum(Lx, Ly, chi, f):
    return sum(f(d0, d1, d2) for d0, d1, d2, _, _, _ in tree(Lx, Ly, chi))


def work(case):
    k = case["kind"]
    if k == "contract":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 16.0 * (M * K + K * N + M * N), "flops": 8.0 * M * N * K}
    Lx, Ly, chi = case["Lx"], case["Ly"], case["chi"]
    if k == "step":
        return _step_work(Lx, Ly, chi)
    size = _node_sum(Lx, Ly, chi, lambda a, b, c: a * b * c)
    if k == "observe":
        # the bond Grams from the root down, two contractions per child leg
        return {"bytes": 16.0 * size,
                "flops": _node_sum(Lx, Ly, chi, lambda a, b, c: 8.0 * a * b * c * (c + a + b))}
    if k == "sample":
        # per shot and node: Gram of child 0 (two contractions), the drawn vector into the node, Gram of child 1
        per = _node_sum(Lx, Ly, chi, lambda a, b, c: 8.0 * (a * b * c * (c + a) + a * b * c + b * c * (c + b) + b * c))
        return {"bytes": 16.0 * size, "flops": per * case["shots"]}
    if k == "compress":
        return {"bytes": 16.0 * (size + _node_sum(Lx, Ly, case["to"], lambda a, b, c: a * b * c)),
                "flops": _node_sum(Lx, Ly, chi, lambda a, b, c: 8.0 * a * b * c * (c + a + b) + 8.0 * 8 * c ** 3)}
    # gradient: the forward steps and, per step, one costate step and one quadrature node's pair of sub-steps
    w = _step_work(Lx, Ly, chi)
    n = case["steps"] * (2 + 2 * case["quad"])
    return {"bytes": w["bytes"] * n, "flops": w["flops"] * n}


# ------------------------------------------------------------------- inputs
def _schedule(case, xy):
    """Pulses of a run: the whole GHZ preparation, or its most parallel CZ layer (minimum CZ distance
    4 a on 8x8, sqrt(8) a elsewhere), repeated so that a long run keeps its drives."""
    Lx, Ly = case["Lx"], case["Ly"]
    r_G = 4.0 if (Lx, Ly) == (8, 8) else math.sqrt(8.0)
    if case.get("pulses", "layer") == "layer":
        rows, T = W.cz_layer_workload(Lx, Ly, r_G)
        again = np.repeat(rows[None], 16, axis=0)
        again[:, :, 1:3] += T * np.arange(16)[:, None, None]
        return again.reshape(-1, 8)
    return W.layers_to_schedule(W.schedule_layers(W.ghz_circuit(Lx, Ly), xy, r_G))[0]


def _product(n, seed):
    """(|0> + e^{i theta}|1>)/sqrt2 on every atom, theta uniform."""
    th = np.random.default_rng(seed).uniform(0.0, 2 * math.pi, n)
    a = np.zeros((n, 3), dtype=np.complex128)
    a[:, 0] = 1.0 / math.sqrt(2.0)
    a[:, 1] = np.exp(1j * th) / math.sqrt(2.0)
    return a


def _entangled(g, seed):
    """Random tree in canonical form: isometric nodes (padding leaves in |0>), a root whose spectrum falls
    from 1 to 1e-6."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    leaf = g.leaf_atoms()
    root = g.num_nodes() - 1
    nodes = []

    def normal(*shape):
        return torch.randn(*shape, dtype=torch.complex128, device="cuda", generator=gen)

    for k in range(root + 1):
        (d0, d1, d2), ch = g.node_info(k)
        if k == root:
            n = min(d0, d1)
            U, V = torch.linalg.qr(normal(d0, n))[0], torch.linalg.qr(normal(d1, n))[0]
            s = 10.0 ** (-6.0 * torch.arange(n, dtype=torch.float64, device="cuda") / max(1, n - 1))
            t = ((U * s) @ V.T).T.reshape(1, d1, d0)
            t = t / torch.linalg.vector_norm(t)
        else:
            a = normal(d1, d0, d2)
            if ch[0] < 0 and leaf[-ch[0] - 1] < 0:
                a[:, 1:] = 0
            if ch[1] < 0 and leaf[-ch[1] - 1] < 0:
                a[1:] = 0
            t = torch.linalg.qr(a.reshape(d1 * d0, d2))[0].T.reshape(d2, d1, d0)
        X = t.contiguous().cpu().numpy().transpose(2, 1, 0)
        g.set_node(k, X)
        nodes.append(t)
    g.refresh_envs()
    return nodes


def _context(case, start, seed):
    Lx, Ly = case["Lx"], case["Ly"]
    xy = W.square_lattice(Lx, Ly)
    g = native.TTN(Lx, Ly, case["chi"])
    g.set_precision(PREC[case.get("prec", "fp64")])
    g.set_hamiltonian(xy, C6)
    if case.get("gamma"):
        g.set_decay(case["gamma"])
    g.apply_pulse(_schedule(case, xy))
    if start == "product":
        g.set_product_state(_product(Lx * Ly, seed))
    else:
        _entangled(g, seed)
    return g


def _segments(case, seed):
    """Two segmented CZ pulses on neighbouring pairs: schedule rows and the differentiated entries."""
    Lx, Ly = case["Lx"], case["Ly"]
    rows, T = W.segmented_cz_schedule([(0, 1), (1, 1 + Lx)], 8, seed)
    rows[:, 1:3] *= DT * case["steps"] / rows[-1, 2]     # the pulses fill the differentiated steps
    params = [(r, f) for r in range(len(rows)) for f in ("omega_r", "delta")]
    return rows, params


def _pair(case, seed):
    """A and B of a contraction as stored (column-major, so B^T-like rows): uniform complex entries."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    M, N, K = case["M"], case["N"], case["K"]

    def u(*shape):
        r = torch.rand(*shape, 2, dtype=torch.float64, device="cuda", generator=gen) * 2 - 1
        return torch.view_as_complex(r)

    return u(K, M), u(N, K)


def prepare(case, seed):
    native.load()
    k = case["kind"]
    st = {"kind": k}
    if k == "contract":
        st["A"], st["B"] = _pair(case, seed)
        st["C"] = torch.empty(case["N"], case["M"], dtype=torch.complex128, device="cuda")
        st["size"] = (case["M"], case["N"], case["K"])
        st["stream"] = torch.cuda.current_stream()
        return st
    if k == "gradient":
        rows, st["params"] = _segments(case, seed)
        g = native.TTN(case["Lx"], case["Ly"], case["chi"])
        g.set_precision(PREC[case["prec"]])
        g.set_hamiltonian(W.square_lattice(case["Lx"], case["Ly"]), C6)
        g.apply_pulse(rows)
        g.set_product_state(_product(g.N, seed))
        st["g"], st["target"] = g, native.TTN(case["Lx"], case["Ly"], case["chi"])
        st["target"].set_ghz([1] * g.N)
        st["steps"], st["quad"] = case["steps"], case["quad"]
        return st
    g = st["g"] = _context(case, case.get("start", "entangled"), seed)
    st["root"], st["split"] = g.num_nodes() - 1, case.get("prec") == "split"
    if k == "observe":
        st["target"] = native.TTN(case["Lx"], case["Ly"], 2)
        st["target"].set_ghz([1] * g.N)
    elif k == "sample":
        st["u"] = np.random.default_rng(seed).random((case["shots"], g.N))
    elif k == "compress":
        st["dst"] = native.TTN(case["Lx"], case["Ly"], case["to"])
    return st


def run(st):
    k = st["kind"]
    if k == "contract":
        M, N, K = st["size"]
        native.contract_split_noalloc(st["A"].data_ptr(), st["B"].data_ptr(), st["C"].data_ptr(), M, N, K,
                                      st["stream"])
        return st["C"]
    g = st["g"]
    if k == "step":
        g.step(DT)
        n, root = g.measure(2), g.get_node(st["root"])
        # split precision contracts in 3xTF32 with FP32 accumulation: what it leaves is kept in single precision
        return {"rydberg": n.astype(np.float32), "root": root.astype(np.complex64)} if st["split"] else \
            {"rydberg": n, "root": root}
    if k == "observe":
        return {"p0": g.measure(0), "rydberg": g.measure(2), "norm": g.norm(),
                "energy": g.energy(), "overlap": np.array([g.overlap(st["target"])])}
    if k == "sample":
        return g.sample(st["u"])
    if k == "compress":
        total, largest = g.compress_into(st["dst"])
        return {"discarded": np.array([total, largest]), "rydberg": st["dst"].measure(2), "norm": st["dst"].norm()}
    F, grad = g.fidelity_gradient(st["target"], DT, st["steps"], st["params"], st["quad"])
    return {"fidelity": F, "gradient": grad}


# ------------------------------------------------- the same in plain 64 bits
SX = np.array([[0, 1, 0], [1, 0, 0], [0, 0, 0]], dtype=np.complex128)
SZ = np.diag([1.0, -1.0, 0.0]).astype(np.complex128)
NR = np.diag([0.0, 0.0, 1.0]).astype(np.complex128)
RP = np.zeros((3, 3), dtype=np.complex128)
RP[2, 1] = 1.0


def _hamiltonian(Lx, Ly, rows, t, gamma):
    """Dense H(t) - i gamma sum n on 3^N states, atom 0 fastest."""
    N = Lx * Ly
    xy = np.array([[i % Lx, i // Lx] for i in range(N)], dtype=np.float64)
    H = np.zeros((3 ** N, 3 ** N), dtype=np.complex128)

    def on(i, op):
        return np.kron(np.eye(3 ** (N - 1 - i)), np.kron(op, np.eye(3 ** i)))

    for i in range(N):
        op = -1j * gamma * NR
        for r in rows:
            if int(r[0]) == i and r[1] <= t < r[2]:
                w = r[5] * np.exp(1j * r[6]) * RP
                op = op + r[3] * SX + r[4] * SZ + w + w.conj().T - r[7] * NR
        H += on(i, op)
    n = [np.real(np.diag(on(i, NR))) for i in range(N)]
    diag = np.zeros(3 ** N)
    for i in range(N):
        for j in range(i + 1, N):
            diag += C6 / np.sum((xy[i] - xy[j]) ** 2) ** 3 * n[i] * n[j]
    return H + np.diag(diag), n


def _expm_apply(H, v, dt):
    """exp(-i dt H) v by its Taylor series in short sub-steps."""
    sub = max(1, int(math.ceil(np.abs(H).sum(1).max() * dt)))
    for _ in range(sub):
        term, k = v, 1
        while np.linalg.norm(term) > 1e-18 * np.linalg.norm(v) and k < 60:
            term = (-1j * dt / sub / k) * (H @ term)
            v = v + term
            k += 1
    return v


def _vector(amps):
    v = np.ones(1, dtype=np.complex128)
    for a in amps:
        v = np.kron(a, v)
    return v


def _exact_tree_observables(case, seed):
    """Populations, norm and GHZ overlap of the tree itself, contracted with torch in complex128."""
    g = native.TTN(case["Lx"], case["Ly"], case["chi"])
    leaf = g.leaf_atoms()
    nodes = _entangled(g, seed)
    info = [g.node_info(k)[1] for k in range(len(nodes))]
    g.close()
    N, root = case["Lx"] * case["Ly"], len(nodes) - 1
    # tensors t[c, b, a]; amp[k]: amplitudes of |0..0> and |1..1> of the subtree in the node's bond basis
    unit = [torch.eye(3, dtype=torch.complex128, device="cuda")[i] for i in range(2)]
    amp = {}
    for k in range(root + 1):
        amp[k] = []
        for s in range(2):
            w = [unit[s if leaf[-c - 1] >= 0 else 0] if c < 0 else amp[c][s] for c in info[k]]
            amp[k].append(torch.einsum("cba,a,b->c", nodes[k], w[0], w[1]))
    overlap = complex((amp[root][0] + amp[root][1]).item()) / math.sqrt(2.0)
    # density of each bond from the root down: rho(a, a') = sum psi(a ..) conj psi(a' ..)
    norm = float(torch.linalg.vector_norm(nodes[root]) ** 2)
    rho, pop = {root: torch.ones(1, 1, dtype=torch.complex128, device="cuda")}, np.zeros((3, N))
    for k in range(root, -1, -1):
        t = nodes[k]
        y = torch.tensordot(rho[k], t, dims=([0], [0]))          # over c: y[c', b, a]
        d = [torch.tensordot(y, t.conj(), dims=([0, 1], [0, 1])), torch.tensordot(y, t.conj(), dims=([0, 2], [0, 2]))]
        for u in range(2):
            c = info[k][u]
            if c >= 0:
                rho[c] = d[u]
            elif leaf[-c - 1] >= 0:
                pop[:, leaf[-c - 1]] = torch.diagonal(d[u]).real.cpu().numpy()
    return {"p0": pop[0], "rydberg": pop[2], "norm": norm, "energy": None,
            "overlap": np.array([overlap])}


def exact(case, seed):
    k = case["kind"]
    if k == "contract":
        A, B = _pair(case, seed)
        return B @ A
    if k == "observe":
        return _exact_tree_observables(case, seed)
    N = case["Lx"] * case["Ly"]
    # a tree whose bonds are complete carries the exact state: every step is the exact exponential
    complete = N <= 6 and case["chi"] >= 3 ** (N // 2)
    if k == "step" and case["start"] == "product" and complete:
        rows = _schedule(case, W.square_lattice(case["Lx"], case["Ly"]))
        H, n = _hamiltonian(case["Lx"], case["Ly"], rows, 0.5 * DT, case["gamma"])
        p = np.abs(_expm_apply(H, _vector(_product(N, seed)), DT)) ** 2
        return {"rydberg": np.array([np.sum(p * x) for x in n]), "root": None}
    if k == "gradient" and complete:
        rows, _ = _segments(case, seed)
        v = _vector(_product(N, seed))
        for i in range(case["steps"]):
            v = _expm_apply(_hamiltonian(case["Lx"], case["Ly"], rows, (i + 0.5) * DT, 0.0)[0], v, DT)
        target = (_vector([[1, 0, 0]] * N) + _vector([[0, 1, 0]] * N)) / math.sqrt(2.0)
        return {"fidelity": float(np.abs(np.vdot(target, v)) ** 2), "gradient": None}
    return None
