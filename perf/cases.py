"""The framework's work as its users have it done, each case through the public calls
of paper_2301_07264_gb300.arso: sampling Pauli errors and running trajectories of one
circuit or of many, the exhaustive single-error analysis, the tolerable-rate search and
the surrogate. Circuits are drawn from the seed; a program holds the compiled circuit,
the criterion and its result buffers, so those are made in prepare().

Scores of complex64 circuits are handed on in 32 bits, which is what that simulation
carries; complex128 circuits keep 64."""
import math

import numpy as np
import torch

from paper_2301_07264_gb300 import arso

SQ = 1.0 / math.sqrt(2.0)


# ---------------------------------------------------------------- circuits --
class Gate:
    def __init__(self, name, *qubits, params=(), matrix=None):
        self.name, self.qubits, self.params, self.matrix = name, qubits, params, matrix


def haar(rng, d):
    z = rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d))
    q, r = np.linalg.qr(z)
    u = q * (np.diag(r) / np.abs(np.diag(r)))
    return u / np.sqrt(np.linalg.det(u)) if d == 2 else u


def toffoli(a, b, c):
    g = Gate
    return [g("H", c), g("CX", b, c), g("TDG", c), g("CX", a, c), g("T", c), g("CX", b, c), g("TDG", c),
            g("CX", a, c), g("T", b), g("T", c), g("H", c), g("CX", a, b), g("T", a), g("TDG", b), g("CX", a, b)]


def mcx(ctrl, tgt, free):
    """Multi-controlled X from Toffolis with borrowed qubits (Barenco et al. 1995, Lemmas 7.2 and 7.3)."""
    m = len(ctrl)
    if m <= 2:
        return [Gate("X", tgt)] if m == 0 else [Gate("CX", ctrl[0], tgt)] if m == 1 else toffoli(ctrl[0], ctrl[1], tgt)
    if len(free) >= m - 2:
        chain = [(ctrl[i + 2], free[i], free[i + 1]) for i in range(m - 3)]
        half = chain[::-1] + [(ctrl[0], ctrl[1], free[0])] + chain
        top = (ctrl[m - 1], free[m - 3], tgt)
        return [g for t in [top] + half + [top] + half for g in toffoli(*t)]
    h = (m + 1) // 2
    low, high = ctrl[:h], ctrl[h:]
    p = mcx(low, free[0], free[1:] + high + [tgt])
    q = mcx(high + [free[0]], tgt, free[1:] + low)
    return p + q + p + q


def circuit(case, rng):
    """(gates, correct outcome or None) of the case's family on n qubits."""
    n, fam, out = case["n"], case["family"], []
    if fam == "brickwork":  # Haar SU(2) on every qubit, CZ on alternating neighbours
        for d in range(case["depth"]):
            out += [Gate("U", q, matrix=haar(rng, 2)) for q in range(n)]
            out += [Gate("CZ", q, q + 1) for q in range(d % 2, n - 1, 2)]
    elif fam == "qaoa":  # two MaxCut layers on a ring with a random chord at every node
        for d in range(2):
            out += [Gate("H", q) for q in range(n)] if d == 0 else []
            ang = rng.uniform(0.0, math.pi, 2)
            for q in range(n):
                for r in ((q + 1) % n, (q + int(rng.integers(2, n))) % n):
                    out += [Gate("CX", q, r), Gate("RZ", r, params=(2 * ang[0],)), Gate("CX", q, r)]
            out += [Gate("RX", q, params=(2 * ang[1],)) for q in range(n)]
    elif fam == "qft":  # of a basis state, swaps as three CX
        out += [Gate("X", q) for q in range(n) if rng.integers(0, 2)]
        for j in range(n - 1, -1, -1):
            out.append(Gate("H", j))
            out += [Gate("CP", k, j, params=(math.pi / (1 << (j - k)),)) for k in range(j - 1, -1, -1)]
        for i in range(n // 2):
            a, b = i, n - 1 - i
            out += [Gate("CX", a, b), Gate("CX", b, a), Gate("CX", a, b)]
    elif fam == "ryrz":  # hardware-efficient ansatz
        for d in range(case["depth"]):
            for q in range(n):
                out += [Gate(k, q, params=(float(rng.uniform(-math.pi, math.pi)),)) for k in ("RY", "RZ")]
            out += [Gate("CX", q, q + 1) for q in range(n - 1)]
    elif fam == "qv":  # quantum volume: Haar U(4) on random pairs
        for _ in range(n):
            p = rng.permutation(n)
            out += [Gate("U2", int(p[2 * k]), int(p[2 * k + 1]), matrix=haar(rng, 4)) for k in range(n // 2)]
    elif fam == "adder":  # ripple carry (Cuccaro et al. 2004) on [c0, b0, a0, ..., z]
        bits = (n - 2) // 2
        a, b = (sum(1 << int(i) for i in rng.permutation(bits)[: (bits + 1) // 2]) for _ in "ab")
        A, B, z = [2 + 2 * i for i in range(bits)], [1 + 2 * i for i in range(bits)], 2 * bits + 1
        out += [Gate("X", A[i]) for i in range(bits) if a >> i & 1] + [Gate("X", B[i]) for i in range(bits) if b >> i & 1]
        prev = [0] + A[:-1]
        for i in range(bits):
            out += [Gate("CX", A[i], B[i]), Gate("CX", A[i], prev[i])] + toffoli(prev[i], B[i], A[i])
        out.append(Gate("CX", A[-1], z))
        for i in reversed(range(bits)):
            out += toffoli(prev[i], B[i], A[i]) + [Gate("CX", A[i], prev[i]), Gate("CX", prev[i], B[i])]
        s = a + b
        right = sum(1 << A[i] for i in range(bits) if a >> i & 1) + sum(1 << B[i] for i in range(bits) if s >> i & 1)
        return out, right + ((s >> bits & 1) << z)
    elif fam == "grover":  # n - 1 search qubits and a borrowed one, in {H, X, CX, T, TDG}
        ns = n - 1
        marked = int(rng.integers(0, 1 << ns))
        search = list(range(ns))
        iters = int(math.pi / (4 * math.asin(2.0 ** (-ns / 2))))
        mcz = [Gate("H", ns - 1)] + mcx(search[:-1], ns - 1, [ns]) + [Gate("H", ns - 1)]
        flip, allx, allh = [Gate("X", q) for q in search if not marked >> q & 1], [Gate("X", q) for q in search], [Gate("H", q) for q in search]
        out = list(allh)
        for _ in range(iters):
            out += flip + mcz + flip + allh + allx + mcz + allx + allh
        return out, marked
    return out, None


def criterion(case, n, right, rng):
    kind = case.get("criterion", "outcome" if right is not None else "fidelity")
    c = {"kind": kind, "threshold": 0.9, "aggregate": "mean" if case["do"] == "exhaustive" else "pass"}
    if kind == "outcome":
        c["target"] = int(rng.integers(0, 1 << n)) if right is None else right
    if kind == "binning":  # half of the outcomes count as success
        c["basis_set"] = tuple(int(v) for v in np.sort(rng.permutation(1 << n)[: 1 << (n - 1)]))
    return c


# ------------------------------------------------------------------- cases --
def listed():
    return [
        # the smallest call: the 4-qubit QFT in double precision, one Monte Carlo estimate of 1,000 trajectories
        {"name": "qft4_c128", "do": "traj", "family": "qft", "n": 4, "precision": 128, "p": 1e-3, "traj": 1000},
        # a sweep of 16 error rates of one deep Clifford+T circuit on chip
        {"name": "grover12_sweep", "do": "sweep", "family": "grover", "n": 12, "rates": 16, "traj": 128},
        # the headline circuit: 24 qubits, 40 layers, on the tiles that the autotuner picks for it
        {"name": "brickwork24", "do": "traj", "family": "brickwork", "n": 24, "depth": 40, "tile": 12, "p": 1e-3, "traj": 200},
        # ordinary streaming circuits on default options, an even and an odd size
        {"name": "brickwork16", "do": "traj", "family": "brickwork", "n": 16, "depth": 40, "p": 1e-3, "traj": 2000},
        {"name": "ryrz17", "do": "traj", "family": "ryrz", "n": 17, "depth": 8, "p": 3e-4, "traj": 777},
        # quantum volume, dense two-qubit gates, scored by the outcomes in a set
        {"name": "qv12", "do": "traj", "family": "qv", "n": 12, "criterion": "binning", "p": 1e-3, "traj": 4000},
        # arithmetic scored by the probability of the right sum
        {"name": "adder20", "do": "traj", "family": "adder", "n": 20, "p": 5e-4, "traj": 500},
        # many circuits of uneven size and family in one call
        {"name": "mix32", "do": "mix", "circuits": 32, "lo": 8, "hi": 22, "p": 5e-4, "traj": 500},
        # Monte Carlo search for the tolerable error rate of one circuit
        {"name": "search14", "do": "search", "family": "brickwork", "n": 14, "depth": 20, "traj": 5000},
        # every single-error state: fidelity, and the probability of the right outcome
        {"name": "exhaustive24", "do": "exhaustive", "family": "brickwork", "n": 24, "depth": 40},
        {"name": "exhaustive_adder20", "do": "exhaustive", "family": "adder", "n": 20},
        # the surrogate: trained on labelled rows, then its predictions over a grid of error rates
        {"name": "surrogate", "do": "surrogate", "rows": 65536, "batch": 8192, "epochs": 1, "grid": 1024},
    ]


def log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["traj", "traj", "traj", "traj", "mix", "sweep", "search", "exhaustive", "exhaustive", "surrogate"])
    p = round(10 ** rng.uniform(-4, -2.5), 7)
    if do == "traj":
        fam = rng.choice(["brickwork", "brickwork", "qaoa", "qft", "ryrz", "qv", "adder"])
        n = rng.randint(10, 16) if fam == "qv" else 2 * rng.randint(3, 11) if fam == "adder" else rng.randint(5, 23)
        c = {"do": do, "family": fam, "n": n, "p": p}
        if fam in ("brickwork", "ryrz"):
            c["depth"] = rng.randint(3, 40)
        if fam != "adder":
            c["criterion"] = rng.choice(["fidelity", "fidelity", "binning" if n <= 18 else "fidelity", "outcome"])
        if n <= 12 and rng.random() < 0.2:
            c["precision"] = 128
        if n >= 15 and rng.random() < 0.3:
            c["tile"] = rng.randint(10, 14)
        gates = sum(span_flops(c)[0].values())
        most = 4.5e12 / (gates * 2.0 ** n * (300 if "precision" in c else 1))
        c["traj"] = max(16, min(log_int(rng, 64, 8000), int(most)))
        return c
    if do == "mix":
        return {"do": do, "circuits": rng.randint(3, 32), "lo": rng.randint(5, 12), "hi": rng.randint(13, 20), "p": p, "traj": log_int(rng, 50, 500)}
    if do == "sweep":
        return {"do": do, "family": rng.choice(["grover", "qaoa", "qft"]), "n": rng.randint(6, 12), "rates": rng.randint(2, 16), "traj": log_int(rng, 16, 128)}
    if do == "search":
        return {"do": do, "family": rng.choice(["brickwork", "qaoa"]), "n": rng.randint(10, 16), "depth": rng.randint(8, 24), "traj": log_int(rng, 500, 5000)}
    if do == "exhaustive":
        fam = rng.choice(["brickwork", "qaoa", "adder"])
        return {"do": do, "family": fam, "n": 2 * rng.randint(3, 11) if fam == "adder" else rng.randint(5, 23), "depth": rng.randint(3, 40)}
    batch = log_int(rng, 500, 16384)
    return {"do": do, "rows": batch * rng.randint(1, 6) + rng.randint(0, batch - 1), "batch": batch, "epochs": rng.randint(1, 2), "grid": log_int(rng, 64, 65536)}


def compiled(case, rng):
    gates, right = circuit(case, rng)
    prec = arso.C128 if case.get("precision") == 128 else arso.C64
    cc = arso.compile_circuit(case["n"], gates, precision=prec, tile_qubits=case.get("tile", 0))
    return gates, cc, criterion(case, case["n"], right, rng)


FAMILIES = ("qft", "qaoa", "adder", "grover", "brickwork", "ryrz")


def mix_members(case):
    """Families in turn over the range of sizes; the deep Grover circuits stay within 10 qubits."""
    out = []
    for i in range(case["circuits"]):
        n = case["lo"] + i * (case["hi"] - case["lo"]) // max(1, case["circuits"] - 1)
        fam = FAMILIES[i % len(FAMILIES)]
        n = min(n, 10) if fam == "grover" else n - n % 2 if fam == "adder" else n
        out.append({"do": "mix", "family": fam, "n": max(n, 4), "depth": 6})
    return out


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    do, dev = case["do"], "cuda"
    st = {"case": case, "seed": int(seed), "stream": torch.cuda.Stream()}
    st["stream"].wait_stream(torch.cuda.current_stream())
    if do == "surrogate":  # rows as the framework labels them: circuit features, log10 p, and a pass flag
        n = case["rows"] + case["grid"]
        x = rng.standard_normal((n, arso.SURROGATE_INPUTS)).astype(np.float32)
        x[:, :10] = np.abs(x[:, :10]) * 30 + 1
        x[:, 10:28] = np.floor(np.abs(x[:, 10:28]) * 20)
        x[:, 32] = rng.uniform(-5, -1, n)
        y = (rng.random(n) < np.exp(-10.0 ** x[:, 32] * 20 * x[:, 0])).astype(np.float32)
        x, y = torch.from_numpy(x).to(dev), torch.from_numpy(y).to(dev)
        st.update(x=x[: case["rows"]].contiguous(), y=y[: case["rows"]].contiguous(), grid=x[case["rows"]:].contiguous(),
                  pred=torch.empty(case["grid"], dtype=torch.float32, device=dev))
        torch.cuda.synchronize()
        return st
    members = mix_members(case) if do == "mix" else [case]
    made = [compiled(m, rng) for m in members]
    st.update(members=members, gates=[m[0] for m in made], cc=[m[1] for m in made], crit=[m[2] for m in made])
    if do == "sweep":
        st["rates"] = np.logspace(-5, -2, case["rates"])
        st["cc"], st["crit"] = st["cc"] * case["rates"], st["crit"] * case["rates"]
    st["c"] = [arso.make_criterion(c) for c in st["crit"]]
    if do in ("traj", "mix", "sweep"):
        st["score"] = [torch.empty(case["traj"], dtype=torch.float64, device=dev) for _ in st["cc"]]
        st["flag"] = torch.empty(case["traj"], dtype=torch.uint8, device=dev)
    torch.cuda.synchronize()
    return st


def run(st):
    case, stream, seed = st["case"], st["stream"], st["seed"]
    do = case["do"]
    with torch.cuda.stream(stream):
        if do == "traj":
            p = case["p"] / 3
            errs = arso.sample_errors(st["cc"][0], p, p, p, seed, 0, case["traj"], stream)
            arso.run_trajectories(st["cc"][0], errs, st["c"][0], st["score"][0], st["flag"], stream)
            mean, passed = arso.aggregate(st["score"][0], st["flag"], stream)[:2]
            wide = case.get("precision") == 128
            out = [st["score"][0] if wide else st["score"][0].float(), float(mean)]
            return out + [float(passed)] if case["family"] == "brickwork" else out
        if do in ("mix", "sweep"):
            p = st["rates"] / 3 if do == "sweep" else case["p"] / 3
            errs = arso.sample_errors_batch(st["cc"], p, p, p, seed, 0, case["traj"], stream)
            arso.run_batch(st["cc"], errs, st["c"], st["score"], None, stream)
            return [s.float() for s in st["score"]]
        if do == "search":
            r = arso.tolerable_rate(st["cc"][0], st["c"][0], 2 / 3, p_lo=1e-5, p_hi=0.1, rel_tol=0.02, n_traj=case["traj"],
                                    seed=seed, mode="mc", stream=stream)
            return [r.p, r.value_lo, r.value_hi]
        if do == "exhaustive":
            P, per = arso.exhaustive(st["cc"][0], st["c"][0], True, stream)
            return [P.astype(np.float32), per.astype(np.float32)]
        s = arso.surrogate_create(seed)
        arso.surrogate_train(s, st["x"], st["y"], epochs=case["epochs"], batch=case["batch"], lr=2e-3, seed=seed, stream=stream)
        arso.surrogate_predict(s, st["grid"], st["pred"], stream)
        return [arso.surrogate_get_params(s), st["pred"]]


# -------------------------------------------------------------------- work --
PER_AMP = {"dense1": 8.0, "diag": 3.0, "h": 2.0, "dense2": 30.0, "perm": 0.0}  # FP32 operations per amplitude


def span_flops(case):
    """({kind: gates}, error locations) of the case's circuit, from its sizes alone."""
    n, fam, d = case["n"], case["family"], case.get("depth", 0)
    if fam == "brickwork":
        return {"dense1": n * d, "perm": (n - 1) * d // 2}, n * d + (n - 1) * d
    if fam == "qaoa":
        return {"dense1": 2 * n, "h": n, "diag": 4 * n, "perm": 8 * n}, 23 * n
    if fam == "qft":
        return {"h": n, "diag": n * n // 2, "perm": 2 * n}, n * n + 4 * n
    if fam == "ryrz":
        return {"dense1": n * d, "diag": n * d, "perm": (n - 1) * d}, 4 * n * d
    if fam == "qv":
        return {"dense2": n * (n // 2)}, n * n
    if fam == "adder":
        return {"h": 2 * n, "diag": 7 * n, "perm": 8 * n}, 25 * n
    g = 5.3 * 15 * n * 2 ** (n / 2)  # Grover: Toffolis of two multi-controlled X an iteration
    return {"h": g * 2 / 15, "diag": g * 7 / 15, "perm": g * 6 / 15}, 1.4 * g


def expected(lam, to_end):
    """(share of trajectories with an error, mean share of the circuit from the first error to the last, or to the end)."""
    if lam > 200:
        return 1.0, 1 - (1 if to_end else 2) / lam
    span, pk = 0.0, math.exp(-lam)
    for k in range(1, int(lam + 12 * math.sqrt(lam) + 20)):
        pk *= lam / k
        span += pk * (k / (k + 1) if to_end else (k - 1) / (k + 1))
    return 1 - math.exp(-lam), span


def traj_work(case, p, traj):
    kinds, L = span_flops(case)
    some, span = expected(L * p, case.get("criterion") == "binning")
    amps = 2.0 ** case["n"]
    flops = traj * span * amps * sum(PER_AMP[k] * v for k, v in kinds.items())
    state = 8.0 * amps * (2 if case.get("precision") == 128 else 1)
    # a state beyond one SM's memory is read where the trajectory restarts and its score reads the reference
    moved = traj * some * 2 * state if case["n"] > 13 else 2 * state
    return {"bytes": moved + 9.0 * traj, "flops": flops}


def work(case):
    do = case["do"]
    if do == "traj":
        return traj_work(case, case["p"], case["traj"])
    if do == "sweep":
        parts = [traj_work(case, p, case["traj"]) for p in np.logspace(-5, -2, case["rates"])]
    elif do == "mix":
        parts = [traj_work(m, case["p"], case["traj"]) for m in mix_members(case)]
    elif do == "search":  # the probes share their errors: about one run at the tolerable rate and one above it
        parts = [traj_work(case, 2e-3, 2 * case["traj"])]
    elif do == "exhaustive":
        kinds, L = span_flops(case)
        states = 2 if case["family"] == "adder" else 1
        amps = 2.0 ** case["n"] * states
        # one sweep: each gate, and for each location the three Pauli expectations of its qubit
        parts = [{"bytes": 16.0 * amps + 24.0 * L, "flops": amps * (sum(PER_AMP[k] * v for k, v in kinds.items()) + 8.0 * L)}]
    else:
        mac = 33 * 256 + 256 * 256 + 256
        parts = [{"bytes": 34 * 4.0 * case["rows"] * case["epochs"] + 34 * 4.0 * case["grid"] + 24.0 * mac,
                  "flops": 2.0 * mac * (3 * case["rows"] * case["epochs"] + case["grid"])}]
    return {k: float(sum(x[k] for x in parts)) for k in ("bytes", "flops")}


# ------------------------------------------------------------------- exact --
def philox(j, t, seed):
    """Philox4x32-10 (Salmon et al., SC'11) of the counters (j, t, t >> 32, 0x41525345) under the seed as key."""
    m = np.uint64(0xFFFFFFFF)
    c = [j.astype(np.uint64), t.astype(np.uint64) & m, t.astype(np.uint64) >> np.uint64(32), np.full_like(j, 0x41525345, dtype=np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for r in range(10):
        a, b = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(b >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), b & m, (a >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), a & m]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def sampled(L, p, traj, seed):
    """Per error location: [(trajectory, Pauli)], with p_X = p_Z = p_Y = p / 3."""
    at = [[] for _ in range(L)]
    third = p / 3
    pt = third + third + third
    thr = min(math.floor(pt * 2.0 ** 32), 2 ** 32 - 1)
    cut = math.floor(third / pt * 2.0 ** 32), math.floor((third + third) / pt * 2.0 ** 32)
    j, t = np.meshgrid(np.arange((L + 1) // 2), np.arange(traj))
    w = philox(j, t, seed)
    for half in (0, 1):
        for tr, pair in zip(*np.nonzero(w[2 * half] < thr)):
            loc = 2 * int(pair) + half
            if loc < L:
                v = int(w[2 * half + 1][tr, pair])
                at[loc].append((int(tr), "X" if v < cut[0] else "Z" if v < cut[1] else "Y"))
    return at


def matrix(g):
    t = g.params[0] if g.params else 0.0
    e = np.exp(1j * np.pi / 4)
    c, s = math.cos(t / 2), math.sin(t / 2)
    one = {"H": [[SQ, SQ], [SQ, -SQ]], "X": [[0, 1], [1, 0]], "Y": [[0, -1j], [1j, 0]], "Z": [[1, 0], [0, -1]], "T": [[1, 0], [0, e]],
           "TDG": [[1, 0], [0, np.conj(e)]], "RX": [[c, -1j * s], [-1j * s, c]], "RY": [[c, -s], [s, c]],
           "RZ": [[np.exp(-0.5j * t), 0], [0, np.exp(0.5j * t)]]}
    if g.matrix is not None:
        return np.asarray(g.matrix)
    if g.name in one:
        return np.asarray(one[g.name], dtype=complex)
    if g.name == "CX":  # local index: control + 2 target
        return np.eye(4, dtype=complex)[[0, 3, 2, 1]]
    return np.diag([1, 1, 1, -1 if g.name == "CZ" else np.exp(1j * t)]).astype(complex)


def applied(psi, n, g, u=None):
    """The gate on every row of psi (rows x 2^n, complex128); local index of two qubits: first + 2 second."""
    u = matrix(g) if u is None else u
    if len(g.qubits) == 1:
        v = psi.view(-1, 2, 1 << g.qubits[0])
        parts = [v[:, 0], v[:, 1]]
    else:
        hi, lo = max(g.qubits), min(g.qubits)
        v = psi.view(-1, 2, 1 << (hi - lo - 1), 2, 1 << lo)
        at = [(0, 0), (0, 1), (1, 0), (1, 1)] if g.qubits[1] == hi else [(0, 0), (1, 0), (0, 1), (1, 1)]
        parts = [v[:, a, :, b] for a, b in at]
    new = torch.empty_like(v)
    for k in range(len(parts)):
        acc = None
        for l in np.nonzero(u[k])[0]:
            acc = complex(u[k][l]) * parts[l] if acc is None else acc.add_(parts[l], alpha=complex(u[k][l]))
        if len(g.qubits) == 1:
            new[:, k] = acc
        else:
            new[:, at[k][0], :, at[k][1]] = acc
    return new.view(psi.shape)


def start(n, rows):
    psi = torch.zeros((rows, 1 << n), dtype=torch.complex128, device="cuda")
    psi[:, 0] = 1
    return psi


def simulated(gates, n, rows, at):
    """Final states of `rows` trajectories; at: per location its [(row, Pauli)]."""
    psi, loc = start(n, rows), 0
    for g in gates:
        psi = applied(psi, n, g)
        for q in g.qubits:
            for kind in "XZY":
                hit = [r for r, k in at[loc] if k == kind]
                if hit:
                    psi[hit] = applied(psi[hit], n, Gate(kind, q))
            loc += 1
    return psi


def scores(psi, ref, crit):
    if crit["kind"] == "fidelity":
        return (psi @ ref.conj()).abs().square()
    if crit["kind"] == "outcome":
        return psi[:, crit["target"]].abs().square()
    return psi[:, torch.tensor(crit["basis_set"], device=psi.device)].abs().square().sum(1)


def exact_scores(gates, n, crit, p, traj, seed):
    at = sampled(sum(len(g.qubits) for g in gates), p, traj, seed)
    rows = sorted({r for a in at for r, _ in a})
    ref = simulated(gates, n, 1, [[]] * len(at))
    out = scores(ref, ref[0], crit).repeat(traj)
    step = max(1, min(1024, (1 << 28) >> n))
    for k in range(0, len(rows), step):
        part = {r: i for i, r in enumerate(rows[k: k + step])}
        psi = simulated(gates, n, len(part), [[(part[r], v) for r, v in a if r in part] for a in at])
        out[list(part)] = scores(psi, ref[0], crit)
    return out


def exact_single(gates, n, crit):
    """Every single-error state's score: <psi|P|psi>^2, or |<phi|P|psi>|^2 with phi carried back from the outcome."""
    psi = start(n, 1)
    for g in gates:
        psi = applied(psi, n, g)
    r = float(scores(psi, psi[0], crit)[0])
    phi = psi.clone()
    if crit["kind"] == "outcome":
        phi = torch.zeros_like(psi)
        phi[0, crit["target"]] = 1
    back = []
    for g in reversed(gates):
        for q in reversed(g.qubits):
            a, b = psi.view(-1, 2, 1 << q), phi.view(-1, 2, 1 << q)
            t = [[(b[:, x].conj() * a[:, y]).sum() for y in (0, 1)] for x in (0, 1)]
            back.append(torch.stack([t[0][1] + t[1][0], t[0][0] - t[1][1], 1j * (t[1][0] - t[0][1])]))
        u = matrix(g).conj().T
        psi, phi = applied(psi, n, g, u), applied(phi, n, g, u)
    per = torch.stack(back[::-1]).abs().square().T.cpu().numpy()
    return np.array([r] + [float(np.mean(v)) for v in per]), per.reshape(-1)


def exact(case, seed):
    do, rng = case["do"], np.random.default_rng(seed)
    if do in ("surrogate", "search", "sweep"):
        return None
    members = mix_members(case) if do == "mix" else [case]
    out = []
    for m in members:
        gates, right = circuit(m, rng)
        crit = criterion(m, m["n"], right, rng)
        if do == "exhaustive":
            if len(gates) * 2.0 ** m["n"] > 3e10:
                return None
            return list(exact_single(gates, m["n"], crit))
        cost = len(gates) * (2.0 ** m["n"] * case["traj"] + 5e5)
        if cost > (1e10 if do == "mix" else 3e11) or len(gates) > 5000:
            out.append(None)
            continue
        out.append(exact_scores(gates, m["n"], crit, case["p"], case["traj"], seed))
    if do == "mix":
        return out
    if out[0] is None:
        return None
    s = out[0]
    got = [s, float(s.mean())]
    return got + [float((s >= 0.9).double().mean())] if case["family"] == "brickwork" else got
