"""The work that users of this library have it do, as cases to be timed.

Each case is one call (or the few calls) that a program makes through the package's public
functions, on inputs made from a seed alone.  Sizes are those of the library's own benchmark,
tests and serving ranges: state vectors of 8 to 30 qubits in both precisions, noisy batches of 1
to 6 qubits, gradients up to 24 qubits, and bursts of circuits through the server.

``exact`` restates each case in plain torch, in 64 bits and gate by gate.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2008_13490_gb300 as qs
from paper_2008_13490_gb300.autograd import circuit_probabilities

K = qs.KIND
SHOTS = 1000


def listed():
    return [
        # The smallest calls: a short circuit on a few qubits, as in a variational loop or an
        # interactive session; latency and launches are all there is.
        {"name": "layered_8q", "kind": "layered", "n": 8, "layers": 10, "prec": "c64", "out": "probs"},
        # Haar layers with CNOTs on random pairs, all outcome probabilities in double precision:
        # the reference workload for one small circuit.
        {"name": "haar_cnot_10q_c128", "kind": "haar_cnot", "n": 10, "layers": 20},
        # An ordinary circuit of the serving range, deep, with an odd number of qubits; the state
        # fits the L2 cache, so planning, uploads and launches weigh as much as the passes.
        {"name": "layered_21q", "kind": "layered", "n": 21, "layers": 60, "prec": "c64", "out": "probs"},
        # The benchmark's headline: 30 qubits, 40 layers, and the whole distribution.
        {"name": "layered_30q", "kind": "layered", "n": 30, "layers": 40, "prec": "c64", "out": "probs"},
        # A Fourier transform of a basis state at the same size: controlled phases and a bit
        # reversal in place of dense layers; the amplitudes stay in the caller's tensor.
        {"name": "qft_30q", "kind": "qft", "n": 30},
        # Double precision at a size where the state is far larger than the caches: the reference
        # runs against which single precision is judged.
        {"name": "layered_25q_c128", "kind": "layered", "n": 25, "layers": 40, "prec": "c128", "out": "state"},
        # Every kind of gate on arbitrary qubits: no locality and no layers, permutations, phases
        # and dense two-qubit gates mixed.
        {"name": "gate_mix_27q", "kind": "gate_mix", "n": 27, "gates": 300},
        # 4096 noisy circuits of 1 to 6 qubits, probabilities and log-likelihoods: scoring a noise
        # model against measured counts.
        {"name": "noisy_4096", "kind": "noisy", "circuits": 4096, "n_max": 6, "len_max": 256, "grad": False},
        # The same with the likelihood's gradient: one step of fitting that model.
        {"name": "noisy_4096_grad", "kind": "noisy", "circuits": 4096, "n_max": 6, "len_max": 256, "grad": True},
        # One training step of a rotation circuit through autograd, parameters in single precision.
        {"name": "train_24q", "kind": "train", "n": 24, "layers": 20},
        # Reading a large state out: its distribution under readout errors, a marginal, every
        # qubit's Bloch vector and the likelihood of counts.
        {"name": "readout_28q", "kind": "readout", "n": 28, "prec": "c64"},
        # A burst of circuits of mixed sizes through the server: small ones packed into the
        # persistent kernel, larger ones on its workers.
        {"name": "serve_24", "kind": "serve", "count": 24, "n_min": 8, "n_max": 26, "d_min": 10, "d_max": 200},
    ]


def draw(rng):
    """One more case of the ranges that the listed ones stand for."""
    kind = rng.choice(["small", "haar_cnot", "layered", "layered", "qft", "layered_c128", "gate_mix", "noisy",
                       "noisy", "train", "readout", "serve"])

    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "small":
        return {"kind": "layered", "n": rng.randint(4, 12), "layers": log(4, 100), "prec": rng.choice(["c64", "c64", "c128"]),
                "out": rng.choice(["probs", "state"])}
    if kind == "haar_cnot":
        return {"kind": "haar_cnot", "n": rng.randint(6, 15), "layers": log(5, 60)}
    if kind == "layered":
        return {"kind": "layered", "n": rng.randint(13, 29), "layers": log(10, 80), "prec": "c64",
                "out": rng.choice(["probs", "state"])}
    if kind == "layered_c128":
        return {"kind": "layered", "n": rng.randint(12, 24), "layers": log(5, 60), "prec": "c128", "out": "state"}
    if kind == "qft":
        return {"kind": "qft", "n": rng.randint(13, 29)}
    if kind == "gate_mix":
        return {"kind": "gate_mix", "n": rng.randint(12, 27), "gates": log(40, 500)}
    if kind == "noisy":
        return {"kind": "noisy", "circuits": log(64, 4096), "n_max": rng.randint(2, 6), "len_max": log(16, 256),
                "grad": rng.random() < 0.5}
    if kind == "train":
        return {"kind": "train", "n": rng.randint(8, 23), "layers": log(3, 20)}
    if kind == "readout":
        return {"kind": "readout", "n": rng.randint(16, 28), "prec": rng.choice(["c64", "c64", "c128"])}
    return {"kind": "serve", "count": rng.randint(6, 24), "n_min": 8, "n_max": rng.randint(13, 25), "d_min": 10,
            "d_max": log(20, 200)}


# ---- circuits as gate records ------------------------------------------------------------------

def _haar(g, count):
    """Haar-random SU(2) matrices [[a, -b*], [b, a*]], from normalised complex Gaussian pairs."""
    v = g.normal(size=(count, 4))
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    a, b = v[:, 0] + 1j * v[:, 1], v[:, 2] + 1j * v[:, 3]
    return np.stack([a, -b.conj(), b, a.conj()], axis=1)


def _records(kinds, q0, q1, mats=None, params=None):
    arr = np.zeros(len(kinds), dtype=qs.GATE_DTYPE)
    arr["kind"], arr["q"][:, 0], arr["q"][:, 1] = kinds, q0, q1
    if mats is not None:
        w = 2 * mats.shape[1]
        arr["m"][:, 0:w:2], arr["m"][:, 1:w:2] = mats.real, mats.imag
    if params is not None:
        arr["param"][:, : params.shape[1]] = params
    return arr


def _haar_layer(g, n):
    return _records(np.full(n, K["MAT1"]), np.arange(n), 0, _haar(g, n))


def _layered(n, layers, g):
    """Haar SU(2) on every qubit, then CZ on alternating neighbour pairs."""
    parts = []
    for layer in range(layers):
        a = np.arange(layer % 2, n - 1, 2)
        parts += [_haar_layer(g, n), _records(np.full(len(a), K["CZ"]), a, a + 1)]
    return np.concatenate(parts)


def _haar_cnot(n, layers, g):
    parts = []
    for _ in range(layers):
        p = g.permutation(n)[: n // 2 * 2].reshape(-1, 2)
        parts += [_haar_layer(g, n), _records(np.full(len(p), K["CNOT"]), p[:, 0], p[:, 1])]
    return np.concatenate(parts)


def _qft(n):
    kinds, q0, q1, ang = [], [], [], []
    for i in range(n - 1, -1, -1):
        kinds.append(K["H"]), q0.append(i), q1.append(0), ang.append(0.0)
        for j in range(i - 1, -1, -1):
            kinds.append(K["CP"]), q0.append(j), q1.append(i), ang.append(2 * math.pi / (1 << (i - j + 1)))
    for i in range(n // 2):
        kinds.append(K["SWAP"]), q0.append(i), q1.append(n - 1 - i), ang.append(0.0)
    return _records(np.array(kinds), np.array(q0), np.array(q1), params=np.array(ang)[:, None])


_MIX1 = ["X", "Y", "Z", "H", "S", "T", "RX", "RY", "RZ", "U1", "U3", "MAT1"]
_MIX2 = ["CNOT", "CZ", "CP", "SWAP", "MAT2"]


def _gate_mix(n, count, g):
    """70 % one-qubit and 30 % two-qubit gates of every kind, on arbitrary qubits."""
    two = g.random(count) < 0.3
    names = np.where(two, np.array(_MIX2)[g.integers(0, len(_MIX2), count)], np.array(_MIX1)[g.integers(0, len(_MIX1), count)])
    q0 = g.integers(0, n, count)
    q1 = np.where(two, (q0 + g.integers(1, n, count)) % n, 0)
    arr = _records(np.array([K[x] for x in names]), q0, q1, params=g.uniform(-math.pi, math.pi, (count, 3)))
    for i in np.nonzero((names == "MAT1") | (names == "MAT2"))[0]:
        d = 2 if names[i] == "MAT1" else 4
        q, r = np.linalg.qr(g.normal(size=(d, d)) + 1j * g.normal(size=(d, d)))
        u = (q * (np.diag(r) / np.abs(np.diag(r)))).reshape(-1)
        arr["m"][i, 0:2 * d * d:2], arr["m"][i, 1:2 * d * d:2] = u.real, u.imag
    return arr


def _rotations(n, layers, g):
    """RX, RY, RZ on every qubit, then CZ on alternating neighbour pairs; angles in float32."""
    parts = []
    for layer in range(layers):
        a = np.arange(layer % 2, n - 1, 2)
        parts += [_records(np.full(n, K[k]), np.arange(n), 0) for k in ("RX", "RY", "RZ")]
        parts.append(_records(np.full(len(a), K["CZ"]), a, a + 1))
    arr = np.concatenate(parts)
    theta = np.zeros((len(arr), 3), dtype=np.float32)
    theta[:, 0] = np.where(arr["kind"] == K["CZ"], 0, g.uniform(-math.pi, math.pi, len(arr)))
    return arr, theta


def _burst(case, seed):
    """(n, gates, mask) of a burst: sizes evenly spread, depths spread by the golden ratio."""
    g = np.random.default_rng([seed, 7])
    out = []
    for i in range(case["count"]):
        n = case["n_min"] + (case["n_max"] - case["n_min"]) * i // max(1, case["count"] - 1)
        depth = case["d_min"] + int((case["d_max"] - case["d_min"]) * ((0.5 + i * 0.6180339887) % 1.0))
        out.append((n, _layered(n, depth, g), (1 << min(n, 10)) - 1))
    return [out[i] for i in np.random.default_rng(7).permutation(len(out))]


# ---- noisy batches -----------------------------------------------------------------------------

def _batch(case, seed):
    """As many circuits of each size 1..n_max, of 1..len_max ops over X90, Y90, CZ and idle, their true
    parameters, the parameters at which a fit stands, and 1000-shot counts at the true ones."""
    g = np.random.default_rng([seed, 4])
    C = case["circuits"]
    nq = g.permutation(np.arange(C) % case["n_max"] + 1).astype(np.int32)
    lens = g.integers(1, case["len_max"] + 1, C)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    n = np.repeat(nq, lens)
    code = g.integers(0, 4, off[-1])
    code = np.where((code == 2) & (n == 1), 0, code)
    a = (g.random(off[-1]) * n).astype(np.int64)
    b = (a + 1 + (g.random(off[-1]) * np.maximum(n - 1, 1)).astype(np.int64)) % np.maximum(n, 2)
    ops = np.stack([code, np.where(code == 3, -1, a), np.where(code == 2, b, -1)], axis=1).astype(np.int32)
    true = np.stack([math.pi / 2 + 0.02 * g.normal(size=C), math.pi / 2 + 0.02 * g.normal(size=C),
                     g.uniform(1e-4, 1e-2, C), g.uniform(1e-4, 1e-2, C)], axis=1)
    at = true.copy()
    at[:, :2] += 0.01 * g.normal(size=(C, 2))
    at[:, 2:] *= g.uniform(0.8, 1.2, size=(C, 2))
    out_off = np.concatenate([[0], np.cumsum(1 << nq.astype(np.int64))]).astype(np.int64)
    batch = SimpleNamespace(size=C, nq=nq, op_off=off, ops=ops, params=true, cnt_off=out_off, counts=None)
    p, _ = _noisy_exact(batch, False)
    p = p.cpu().numpy()
    counts = np.zeros(out_off[-1], dtype=np.int32)
    for k in range(1, case["n_max"] + 1):
        which = np.nonzero(nq == k)[0]
        if len(which):
            at_k = out_off[which][:, None] + np.arange(1 << k)
            # rounded, so that the draw does not hang on the last bits of the sums above
            w = np.round(np.clip(p[at_k], 0, None), 9)
            counts[at_k] = g.multinomial(SHOTS, w / w.sum(axis=1, keepdims=True))
    batch.params, batch.counts = at, counts
    return batch


def _digit(x, M, q):
    """4x4 matrices M [C, 4, 4] on base-4 digit q of x [C, T, 4^n]."""
    C, T, D = x.shape
    b = 4 ** q
    return torch.matmul(M[:, None], x.reshape(C, T * (D // (4 * b)), 4, b)).reshape(C, T, D)


def _noisy_exact(batch, tangents, dev=None):
    """Probabilities [out_off[-1]] and, with `tangents`, their derivatives by the four parameters
    [4, out_off[-1]], in 64 bits: every circuit's Pauli vector, all circuits of one size together."""
    dev = dev or ("cuda" if torch.cuda.is_available() else "cpu")
    f8 = {"dtype": torch.float64, "device": dev}
    P = torch.zeros(int(batch.cnt_off[-1]), **f8)
    dP = torch.zeros((4, int(batch.cnt_off[-1])), **f8) if tangents else None
    for n in range(1, int(batch.nq.max()) + 1):
        which = np.nonzero(batch.nq == n)[0]
        C, D = len(which), 4 ** n
        if not C:
            continue
        lens = batch.op_off[which + 1] - batch.op_off[which]
        L = int(lens.max())
        ops = np.full((C, L, 3), -1, dtype=np.int64)  # code -1: no op
        rows = np.arange(L)[None] < lens[:, None]
        ops[rows] = batch.ops[(batch.op_off[which][:, None] + np.arange(L))[rows]]
        pars = torch.tensor(batch.params[which], **f8)
        tx, ty, p, gm = pars.T
        one, zero = torch.ones(C, **f8), torch.zeros(C, **f8)

        def mat(rows_):
            return torch.stack([torch.stack(r, dim=1) for r in rows_], dim=1)

        s, k = torch.sqrt(1 - gm), 1 - 4 * p / 3
        ad = mat([[one, zero, zero, zero], [zero, s, zero, zero], [zero, zero, s, zero], [gm, zero, zero, 1 - gm]])
        dad = mat([[zero] * 4, [zero, -0.5 / s, zero, zero], [zero, zero, -0.5 / s, zero], [one, zero, zero, -one]])
        dep = mat([[one, zero, zero, zero], [zero, k, zero, zero], [zero, zero, k, zero], [zero, zero, zero, k]])
        ddep = -4.0 / 3 * torch.diag(torch.tensor([0.0, 1, 1, 1], **f8)).expand(C, 4, 4)
        cx, sx, cy, sy = torch.cos(tx), torch.sin(tx), torch.cos(ty), torch.sin(ty)
        rx = mat([[one, zero, zero, zero], [zero, one, zero, zero], [zero, zero, cx, -sx], [zero, zero, sx, cx]])
        drx = mat([[zero] * 4, [zero] * 4, [zero, zero, -sx, -cx], [zero, zero, cx, -sx]])
        ry = mat([[one, zero, zero, zero], [zero, cy, zero, sy], [zero, zero, one, zero], [zero, -sy, zero, cy]])
        dry = mat([[zero] * 4, [zero, -sy, zero, cy], [zero] * 4, [zero, -cy, zero, -sy]])
        ch, eye, nil = ad @ dep, torch.eye(4, **f8).expand(C, 4, 4), torch.zeros((C, 4, 4), **f8)
        dch = [nil, nil, ad @ ddep, dad @ dep]
        # 0: nothing, 1: the channel, 2: X90 and the channel, 3: Y90 and the channel
        M = torch.stack([eye, ch, ch @ rx, ch @ ry], dim=1)
        dM = torch.stack([torch.stack([nil, dch[j], dch[j] @ rx + (ch @ drx if j == 0 else 0), dch[j] @ ry + (ch @ dry if j == 1 else 0)], dim=1)
                          for j in range(4)], dim=1)  # [C, parameter, choice, 4, 4]
        # CZ on digits (a, b): I/z on one qubit leave the other alone, x/y put a z on it
        idx = np.arange(D)
        zflip = np.array([3, 2, 1, 0])  # the digit that z makes of I, x, y, z
        src, sgn = [idx], [np.ones(D)]
        pair = {}
        for a in range(n):
            for b in range(n):
                if a < b:
                    da, db = idx >> (2 * a) & 3, idx >> (2 * b) & 3
                    xa, xb = (da == 1) | (da == 2), (db == 1) | (db == 2)
                    na, nb = np.where(xb, zflip[da], da), np.where(xa, zflip[db], db)
                    neg = ((da == 1) & (db == 2)) | ((da == 2) & (db == 1))
                    pair[a, b] = pair[b, a] = len(src)
                    src.append(idx + ((na - da) << (2 * a)) + ((nb - db) << (2 * b)))
                    sgn.append(np.where(neg, -1.0, 1.0))
        src, sgn = torch.tensor(np.stack(src), device=dev), torch.tensor(np.stack(sgn), **f8)
        lut = np.zeros((max(n, 1), max(n, 1)), dtype=np.int64)
        for (a, b), v in pair.items():
            lut[a, b] = v
        code, a, b = ops[..., 0], ops[..., 1], ops[..., 2]
        cz = torch.tensor(np.where(code == 2, lut[np.maximum(a, 0), np.maximum(b, 0)], 0), device=dev)
        choice = np.zeros((C, L, n), dtype=np.int64)
        for q in range(n):
            choice[..., q] = np.where(code == 3, 1, np.where((code == 2) & ((a == q) | (b == q)), 1, np.where((code == 0) & (a == q), 2, np.where((code == 1) & (a == q), 3, 0))))
        choice = torch.tensor(choice, device=dev)
        T = 5 if tangents else 1
        r = torch.zeros((C, T, D), **f8)
        zero_state = torch.tensor([1.0, 0, 0, 1], **f8)
        v = torch.ones(1, **f8)
        for _ in range(n):
            v = torch.kron(v, zero_state)
        r[:, 0] = v * 2.0 ** (-n / 2)
        every = torch.arange(C, device=dev)
        for step in range(L):
            if n > 1:
                z = cz[:, step]
                r = torch.gather(r, 2, src[z][:, None].expand(C, T, D)) * sgn[z][:, None]
            for q in range(n):
                c = choice[:, step, q]
                new = _digit(r, M[every, c], q)
                if tangents:
                    x = r[:, :1]
                    for j in range(4):
                        new[:, 1 + j] += _digit(x, dM[every, j, c], q)[:, 0]
                r = new
        # outcome J: sum over I/z digits with the sign of the bits that z meets
        J = np.arange(1 << n)
        iz = sum(((J >> q & 1) * 3) << (2 * q) for q in range(n))
        par = np.array([[(-1.0) ** bin(i & j).count("1") for i in J] for j in J]) * 2.0 ** (-n / 2)
        out = r[:, :, torch.tensor(iz, device=dev)] @ torch.tensor(par, **f8).T
        at = torch.tensor(batch.cnt_off[which][:, None] + J, device=dev)
        P[at] = out[:, 0]
        if tangents:
            for j in range(4):
                dP[j][at] = out[:, 1 + j]
    return P, dP


# ---- preparation, one pass, work ---------------------------------------------------------------

def _prec(case):
    return qs.QS_C128 if case.get("prec") == "c128" else qs.QS_C64


def _circuit(case, seed):
    g = np.random.default_rng([seed, 1])
    kind = case["kind"]
    if kind == "layered":
        return _layered(case["n"], case["layers"], g)
    if kind == "haar_cnot":
        return _haar_cnot(case["n"], case["layers"], g)
    if kind == "gate_mix":
        return _gate_mix(case["n"], case["gates"], g)
    return _qft(case["n"])


def _basis(case, seed):
    return int(np.random.default_rng([seed, 2]).integers(0, 1 << case["n"])) if case["kind"] == "qft" else 0


def _random_state(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    real = torch.float64 if case["prec"] == "c128" else torch.float32
    a = torch.randn(2 << case["n"], dtype=real, device="cuda", generator=gen)
    a /= torch.linalg.vector_norm(a, dtype=torch.float64).to(real)
    return torch.view_as_complex(a.view(-1, 2))


def _readout_inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    counts = torch.randint(0, 3, (1 << case["n"],), dtype=torch.int32, device="cuda", generator=gen)
    g = np.random.default_rng([seed, 3])
    return counts, g.uniform(0.005, 0.08, case["n"]), g.uniform(0.005, 0.08, case["n"])


def _train_inputs(case, seed):
    g = np.random.default_rng([seed, 5])
    gates, theta = _rotations(case["n"], case["layers"], g)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    weights = torch.randn(1 << case["n"], dtype=torch.float64, device="cuda", generator=gen)
    return gates, theta, weights


def prepare(case, seed):
    kind = case["kind"]
    s = SimpleNamespace(case=case)
    if kind in ("layered", "haar_cnot", "qft", "gate_mix"):
        n = case["n"]
        s.gates, s.basis = _circuit(case, seed), _basis(case, seed)
        s.double = kind == "haar_cnot" or case.get("prec") == "c128"
        s.want_probs = kind == "haar_cnot" or case.get("out") == "probs"
        s.amps = torch.zeros(1 << n, dtype=torch.complex128 if s.double else torch.complex64, device="cuda")
        s.state = qs.sv_wrap(s.amps)
        if s.want_probs:
            s.probs = torch.empty(1 << n, dtype=torch.float64 if s.double else torch.float32, device="cuda")
    elif kind == "noisy":
        s.batch = qs.NoisyBatchDevice(_batch(case, seed))
    elif kind == "train":
        s.gates, theta, s.weights = _train_inputs(case, seed)
        s.theta = torch.tensor(theta, requires_grad=True)
    elif kind == "readout":
        s.amps = _random_state(case, seed)
        s.state = qs.sv_wrap(s.amps)
        s.counts, s.e01, s.e10 = _readout_inputs(case, seed)
        s.probs = torch.empty(1 << case["n"], dtype=s.amps.real.dtype, device="cuda")
    else:
        s.jobs = _burst(case, seed)
        s.server = qs.Server(mem_budget=8 << 30)
    return s


def run(s):
    kind = s.case["kind"]
    if kind in ("layered", "haar_cnot", "qft", "gate_mix"):
        qs.sv_set_basis(s.state, s.basis)
        qs.sv_apply_circuit(s.state, s.gates)
        if not s.want_probs:
            return s.amps
        p, _ = qs.sv_probs(s.state, out=s.probs, fp64=s.double, want_norm=False)
        return p
    if kind == "noisy":
        # likelihoods and gradients as a fit that keeps its parameters in float32 takes them
        p, ll, g = s.batch.run(grad=s.case["grad"])
        return {"probs": p, "loglik": ll.float(), "grad": g.float()} if g is not None else {"probs": p, "loglik": ll.float()}
    if kind == "train":
        p = circuit_probabilities(s.theta, s.case["n"], s.gates)
        loss = (p * s.weights).sum()
        (grad,) = torch.autograd.grad(loss, s.theta)
        return {"loss": loss.detach().float(), "grad": grad}
    if kind == "readout":
        real = np.float64 if s.case["prec"] == "c128" else np.float32
        qs.sv_probs(s.state, out=s.probs, fp64=real is np.float64, want_norm=False)
        marginal, _ = qs.sv_probs(s.state, fp64=real is np.float64, marg_mask=(1 << 10) - 1, want_norm=False)
        bloch = qs.sv_bloch(s.state).astype(real)
        loglik, _ = qs.sv_loglik(s.state, s.counts)
        qs.meas_error(s.probs, s.e01, s.e10)
        return {"probs": s.probs, "marginal": marginal, "bloch": bloch, "loglik": float(loglik)}
    # the states are complex64: results are worth 32 bits
    tickets = [s.server.submit(n, gates, mask) for n, gates, mask in s.jobs]
    return [s.server.wait(t)[0].astype(np.float32) for t in tickets]


def _circuit_flops(gates, n):
    """Real operations of a gate list, gate by gate: 14 an amplitude for a dense 2x2, 30 for a
    4x4, 3 for a phase on half of the amplitudes, none for moves and signs."""
    k = gates["kind"]
    free = np.isin(k, [K[x] for x in ("I", "X", "Y", "Z", "S", "SDG", "CNOT", "CZ", "SWAP")])
    phase = np.isin(k, [K[x] for x in ("T", "TDG", "U1", "RK", "CP")])
    per = np.where(free, 0, np.where(phase, 3, np.where(k == K["MAT2"], 30, 14)))
    return float(per.sum()) * 2.0 ** n


def work(case):
    kind = case["kind"]
    if kind in ("layered", "haar_cnot", "qft", "gate_mix"):
        amp = 16 if kind == "haar_cnot" or case.get("prec") == "c128" else 8
        probs = amp / 2 if kind == "haar_cnot" or case.get("out") == "probs" else 0
        return {"bytes": 2.0 ** case["n"] * (amp + probs), "flops": _circuit_flops(_circuit(case, 0), case["n"])}
    if kind == "noisy":
        # a one-qubit op is 4^n multiply-adds of its 7 entries over 4 places, a CZ or an idle
        # step the 5 entries of each qubit's channel; the gradient goes back through each once
        C, L = case["circuits"], (case["len_max"] + 1) / 2
        per = sum(4.0 ** n * (0.5 * 14 + 0.25 * 2 * 10 + 0.25 * n * 10) / 4 for n in range(1, case["n_max"] + 1)) / case["n_max"]
        outs = sum(2.0 ** n for n in range(1, case["n_max"] + 1)) / case["n_max"]
        return {"bytes": C * (L * 16 + outs * 8 + 32 + 8 + (32 if case["grad"] else 0)), "flops": C * L * per * (4 if case["grad"] else 1)}
    if kind == "train":
        n, layers = case["n"], case["layers"]
        f = 2.0 ** n * n * layers * (4 + 4 + 6)
        return {"bytes": 2.0 ** n * (8 + 8 + 8), "flops": 4 * f}
    if kind == "readout":
        n, amp = case["n"], 16 if case["prec"] == "c128" else 8
        return {"bytes": 2.0 ** n * (amp + 4 + amp / 2), "flops": 2.0 ** n * (3 + 8 * n + 3 * n)}
    burst = _burst(case, 0)
    return {"bytes": sum(8.0 * 2 ** n for n, _, _ in burst), "flops": sum(_circuit_flops(gates, n) for n, gates, _ in burst)}


# ---- the same in 64 bits, gate by gate ---------------------------------------------------------

MOST = 2.0e11  # amplitudes times gates: about ten seconds
_S = math.sqrt(0.5)
_ONE = {"I": [[1, 0], [0, 1]], "X": [[0, 1], [1, 0]], "Y": [[0, -1j], [1j, 0]], "Z": [[1, 0], [0, -1]], "H": [[_S, _S], [_S, -_S]],
        "S": [[1, 0], [0, 1j]], "T": [[1, 0], [0, complex(_S, _S)]]}
_NAME = {v: k for k, v in K.items()}


def _matrix(g):
    """The matrix of one gate record, first listed qubit most significant."""
    name, (t, phi, lam) = _NAME[int(g["kind"])], (float(x) for x in g["param"])
    if name in _ONE:
        return np.array(_ONE[name], dtype=complex)
    if name in ("MAT1", "MAT2"):
        d = 2 if name == "MAT1" else 4
        return (g["m"][0:2 * d * d:2] + 1j * g["m"][1:2 * d * d:2]).reshape(d, d)
    c, s = math.cos(t / 2), math.sin(t / 2)
    if name == "RX":
        return np.array([[c, -1j * s], [-1j * s, c]])
    if name == "RY":
        return np.array([[c, -s], [s, c]], dtype=complex)
    if name == "RZ":
        return np.diag([complex(c, -s), complex(c, s)])
    if name == "U1":
        return np.diag([1, np.exp(1j * t)])
    if name == "U3":
        return np.array([[c, -np.exp(1j * lam) * s], [np.exp(1j * phi) * s, np.exp(1j * (phi + lam)) * c]])
    two = {"CZ": np.diag([1, 1, 1, -1]).astype(complex), "CP": np.diag([1, 1, 1, np.exp(1j * t)]),
           "CNOT": np.eye(4, dtype=complex)[[0, 1, 3, 2]], "SWAP": np.eye(4, dtype=complex)[[0, 2, 1, 3]]}
    return two[name]


def _slices(x, n, qubits):
    """The amplitudes of x by the values of `qubits`: views, the first listed most significant."""
    out = []
    order = sorted(qubits, reverse=True)
    shape, top = [], n
    for q in order:
        shape += [1 << (top - q - 1), 2]
        top = q
    v = x.view(shape + [1 << top])
    for val in range(1 << len(qubits)):
        at = [slice(None)] * (2 * len(order) + 1)
        for i, q in enumerate(qubits):
            at[2 * order.index(q) + 1] = val >> (len(qubits) - 1 - i) & 1
        out.append(v[tuple(at)])
    return out


def _apply(x, n, qubits, U):
    d = U.shape[0]
    parts = _slices(x, n, qubits)
    rows = [i for i in range(d) if U[i, i] != 1 or np.count_nonzero(U[i]) > 1]
    old = {j: parts[j].clone() for j in range(d) if any(U[i, j] != 0 and i != j for i in rows)}
    for i in rows:
        terms = [j for j in range(d) if U[i, j] != 0]
        new = None
        for j in terms:
            t = old.get(j, parts[j]) * complex(U[i, j])
            new = t if new is None else new.add_(t)
        parts[i].copy_(new)


def _qubits(g):
    return [int(g["q"][0])] if int(g["kind"]) < K["CNOT"] else [int(g["q"][0]), int(g["q"][1])]


def _evolve(gates, n, basis=0, dev=None):
    x = torch.zeros(1 << n, dtype=torch.complex128, device=dev or ("cuda" if torch.cuda.is_available() else "cpu"))
    x[basis] = 1
    for g in gates:
        _apply(x, n, _qubits(g), _matrix(g))
    return x


def _probs(x):
    return x.real ** 2 + x.imag ** 2


def _marginal(p, k):
    return p.view(-1, 1 << k).sum(dim=0)


def _train_exact(gates, theta, weights, n):
    gates = gates.copy()
    gates["param"] = theta.astype(np.float64)
    x = _evolve(gates, n, dev=weights.device)
    loss = (_probs(x) * weights).sum()
    lam = x * weights
    grad = torch.zeros(len(gates), dtype=torch.float64, device=weights.device)
    for i in range(len(gates) - 1, -1, -1):
        q, U = _qubits(gates[i]), _matrix(gates[i])
        name = _NAME[int(gates[i]["kind"])]
        if name in ("RX", "RY", "RZ"):  # dU/dt = -i/2 sigma U: 2 Re <lam| dU |before> = Im <lam| sigma |after>
            x0, x1 = _slices(x, n, q)
            l0, l1 = _slices(lam, n, q)
            if name == "RZ":
                v = (l0.conj() * x0).sum() - (l1.conj() * x1).sum()
            else:
                v = (l0.conj() * x1).sum() * (1 if name == "RX" else -1j) + (l1.conj() * x0).sum() * (1 if name == "RX" else 1j)
            grad[i] = v.imag
        _apply(x, n, q, U.conj().T)
        _apply(lam, n, q, U.conj().T)
    out = torch.zeros((len(gates), 3), dtype=torch.float64, device=weights.device)
    out[:, 0] = grad
    return loss, out


def exact(case, seed):
    kind = case["kind"]
    if kind == "qft":
        n, J = case["n"], _basis(case, seed)
        k = torch.arange(1 << n, dtype=torch.int64, device="cuda") * J % (1 << n)
        angle = k.to(torch.float64) * (2 * math.pi / (1 << n))
        return torch.polar(torch.full_like(angle, 2.0 ** (-n / 2)), angle)
    if kind in ("layered", "haar_cnot", "gate_mix"):
        gates, n = _circuit(case, seed), case["n"]
        if len(gates) * 2.0 ** n > MOST:
            return None
        x = _evolve(gates, n)
        return _probs(x) if kind == "haar_cnot" or case.get("out") == "probs" else x
    if kind == "noisy":
        batch = _batch(case, seed)
        P, dP = _noisy_exact(batch, case["grad"])
        counts = torch.tensor(batch.counts, dtype=torch.float64, device=P.device)
        owner = torch.tensor(np.repeat(np.arange(batch.size), 1 << batch.nq.astype(np.int64)), device=P.device)

        def per_circuit(v):
            return torch.zeros(batch.size, dtype=torch.float64, device=P.device).index_add_(0, owner, torch.where(counts > 0, v, torch.zeros_like(v)))

        out = {"probs": P, "loglik": per_circuit(counts * torch.log(P.clamp_min(1e-300)))}
        if case["grad"]:
            out["grad"] = torch.stack([per_circuit(counts * dP[j] / P.clamp_min(1e-300)) for j in range(4)], dim=1)
        return out
    if kind == "train":
        gates, theta, weights = _train_inputs(case, seed)
        if len(gates) * 2.0 ** case["n"] > MOST / 4:
            return None
        loss, grad = _train_exact(gates, theta, weights, case["n"])
        return {"loss": loss, "grad": grad}
    if kind == "readout":
        n, x = case["n"], _random_state(case, seed).to(torch.complex128)
        counts, e01, e10 = _readout_inputs(case, seed)
        p = _probs(x)
        marginal = _marginal(p, 10)
        loglik = (torch.where(counts > 0, torch.log(p.clamp_min(1e-300)), torch.zeros_like(p)) * counts).sum()
        bloch = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
        for q in range(n):
            x0, x1 = _slices(x, n, [q])
            v = 2 * (x0.conj() * x1).sum()
            bloch[q, 0], bloch[q, 1], bloch[q, 2] = v.real, v.imag, _probs(x0).sum() - _probs(x1).sum()
        for q in range(n):
            p0, p1 = _slices(p, n, [q])
            a, b = p0 * (1 - e01[q]) + p1 * e10[q], p0 * e01[q] + p1 * (1 - e10[q])
            p0.copy_(a), p1.copy_(b)
        return {"probs": p, "marginal": marginal, "bloch": bloch, "loglik": loglik}
    out, left = [], MOST
    for n, gates, mask in _burst(case, seed):
        cost = len(gates) * 2.0 ** n + 1e7 * len(gates)  # small states cost a launch each
        if cost > left or n > 20:
            out.append(None)
            continue
        left -= cost
        out.append(_marginal(_probs(_evolve(gates, n)), min(n, 10)))
    return out
