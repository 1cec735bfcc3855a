"""The work whose speed counts: calls that users of this library make, from the smallest
circuits to a saturated layer at bond dimension 256, each through the public entry points.

Kinds of case:
  circuit     a whole small program: create a state, run a circuit, read every amplitude;
  gateset     a wide, shallow circuit of the gate set {H, CX, RZZ, RX}: small bonds, many
              small calls, amplitudes of a batch of bitstrings at the end;
  two_site    one two-qubit update on the caller's own device buffers;
  layer       one layer of a Haar SU(4) brickwork on a saturated state (even and odd layers
              in turn), with the entanglement spectra of the bonds that it updated;
  batch       a step of many independent circuits of uneven width and bond dimension, both
              of its layers replayed as one CUDA graph;
  amplitudes  <x|psi> of a batch of bitstrings;
  expect      the Pauli terms of a transverse-field Ising Hamiltonian;
  sample      perfect sampling;
  grad        energy and angle gradient of a hardware-efficient ansatz.

Results of complex64 states are returned in 32 bits, the precision they are computed in
(the entry points widen them).  Site tensors of an updated state are only defined up to
the gauge of their bonds, so a layer returns its gauge-free results: every discarded
weight, bond dimension and kept singular value; the two-site case returns its block.
"""
import numpy as np
import torch

import paper_2601_04422_gb300 as T
import workloads as W

# Sites of a saturated random state: complex Gaussian tensors, as the single-gate samples of
# the benchmark use.  Their gated blocks have the flat, full-rank spectrum of a saturated
# Haar brickwork (6-7 % of the weight discarded at half rank).


def _caps(n, chi):
    return [min(chi, 1 << min(b, n - b, 30)) for b in range(n + 1)]


def _gauss_sites(n, chi, rng, single):
    c = _caps(n, chi)
    sites = []
    for q in range(n):
        shape = (c[q], 2, c[q + 1])
        a = rng.standard_normal(shape + (2,), dtype=np.float32)
        a *= np.float32(1.0 / np.sqrt(4.0 * c[q + 1]))
        a = a.view(np.complex64)[..., 0].astype(np.complex128)
        if not single:   # values that single precision cannot hold
            a *= 1.0 + 1e-9 * rng.standard_normal()
        sites.append(a)
    return sites


def _saturated(case, rng, stream=None):
    single = case["dtype"] == "c64"
    m = T.MPS(case["n"], dtype=T.TNSIM_C64 if single else T.TNSIM_C128, chi_max=case["chi"],
              cutoff=case.get("cutoff", 0.0), gemm=_GEMM[case.get("gemm", "fp32")], stream=stream)
    m.import_sites(_gauss_sites(case["n"], case["chi"], rng, single))
    return m


_GEMM = {"fp32": T.TNSIM_GEMM_FP32, "fp32_3m": T.TNSIM_GEMM_FP32_3M, "tf32x3": T.TNSIM_GEMM_TF32X3,
         "bf16x3": T.TNSIM_GEMM_BF16X3}
_FORM = {"paper": T.TNSIM_FORM_PAPER, "canonical": T.TNSIM_FORM_CANONICAL}


def listed():
    return [
        # the smallest whole program: the exact 10-qubit circuit in the paper's precision
        {"name": "circuit_c128_10q", "kind": "circuit", "n": 10, "depth": 8, "chi": 32, "dtype": "c128",
         "form": "paper", "ops": 0},
        # 100 qubits of the paper's gate set: bonds stay small, launches and calls count
        {"name": "gateset_c128_100q", "kind": "gateset", "n": 100, "depth": 12, "chi": 256, "strings": 64},
        # one gate of a plugin that owns its device memory, at an odd bond dimension
        {"name": "two_site_c64_chi61", "kind": "two_site", "l": 61, "m": 61, "r": 61, "chi": 61},
        # default parameters (chi_max 64, FP32 contraction), a chain of 24 qubits
        {"name": "layer_c64_chi64_24q", "kind": "layer", "n": 24, "chi": 64, "dtype": "c64", "gemm": "fp32",
         "cfg": 0, "cutoff": 0.0},
        # the 64-qubit brickwork: chi_max 128 with a cutoff, tensor-core contraction and
        # the Jacobi configuration that the autotuner picks
        {"name": "layer_c64_chi128_64q", "kind": "layer", "n": 64, "chi": 128, "dtype": "c64", "gemm": "tf32x3",
         "cfg": 2, "cutoff": 1e-10},
        # the benchmark's layer: 100 qubits at chi_max 256
        {"name": "layer_c64_chi256_100q", "kind": "layer", "n": 100, "chi": 256, "dtype": "c64", "gemm": "tf32x3",
         "cfg": 2, "cutoff": 0.0},
        # the paper's precision, a bond dimension off the powers of two
        {"name": "layer_c128_chi90_40q", "kind": "layer", "n": 40, "chi": 90, "dtype": "c128", "gemm": "fp32",
         "cfg": 0, "cutoff": 0.0},
        # many independent circuits of uneven size, as one CUDA graph
        {"name": "batch_c64_16x", "kind": "batch", "states": 16, "n_max": 96, "chi_max": 64, "gemm": "fp32"},
        # read-out of a saturated state: amplitudes for cross-entropy, energies, samples
        {"name": "amplitudes_c64_chi256", "kind": "amplitudes", "n": 100, "chi": 256, "dtype": "c64",
         "strings": 1024},
        {"name": "expect_c64_chi64", "kind": "expect", "n": 50, "chi": 64, "dtype": "c64"},
        {"name": "sample_c64_chi128", "kind": "sample", "n": 64, "chi": 128, "dtype": "c64", "shots": 1024},
        # one step of a variational optimisation
        {"name": "grad_c128_30q", "kind": "grad", "n": 30, "layers": 8, "chi": 64, "cutoff": 1e-6},
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["circuit", "gateset", "two_site", "layer", "layer", "layer", "batch", "amplitudes",
                       "expect", "sample", "grad"])
    if kind == "circuit":
        ops = rng.choice([0, _log_int(rng, 8, 40)])
        return {"kind": kind, "n": rng.randint(4, 12), "depth": rng.randint(2, 10), "chi": 64,
                "dtype": rng.choice(["c64", "c128"]), "form": rng.choice(["paper", "canonical"]), "ops": ops}
    if kind == "gateset":
        return {"kind": kind, "n": _log_int(rng, 12, 100), "depth": rng.randint(3, 12), "chi": 256,
                "strings": _log_int(rng, 1, 256)}
    if kind == "two_site":
        c = [_log_int(rng, 2, 128) for _ in range(3)]
        c[1] = min(c[1], 2 * c[0], 2 * c[2])
        return {"kind": kind, "l": c[0], "m": c[1], "r": c[2], "chi": max(1, min(c[0], c[2], 128))}
    if kind == "layer":
        dtype = rng.choice(["c64", "c64", "c64", "c128"])
        chi = _log_int(rng, 8, 256 if dtype == "c64" else 96)
        return {"kind": kind, "n": _log_int(rng, 16, 100 if dtype == "c64" else 40), "chi": chi, "dtype": dtype,
                "gemm": rng.choice(["fp32", "fp32_3m", "tf32x3", "bf16x3"]) if dtype == "c64" else "fp32",
                "cfg": rng.choice([0, 2]), "cutoff": rng.choice([0.0, 1e-10])}
    if kind == "batch":
        return {"kind": kind, "states": _log_int(rng, 2, 16), "n_max": _log_int(rng, 17, 96),
                "chi_max": rng.choice([16, 32, 64]), "gemm": rng.choice(["fp32", "tf32x3"])}
    if kind == "amplitudes":
        return {"kind": kind, "n": _log_int(rng, 16, 100), "chi": _log_int(rng, 16, 256),
                "dtype": rng.choice(["c64", "c64", "c128"]), "strings": _log_int(rng, 1, 512)}
    if kind == "expect":
        return {"kind": kind, "n": _log_int(rng, 8, 50), "chi": _log_int(rng, 8, 128),
                "dtype": rng.choice(["c64", "c64", "c128"])}
    if kind == "sample":
        return {"kind": kind, "n": _log_int(rng, 10, 100), "chi": _log_int(rng, 8, 128),
                "dtype": rng.choice(["c64", "c64", "c128"]), "shots": _log_int(rng, 1, 1024)}
    return {"kind": kind, "n": _log_int(rng, 6, 30), "layers": rng.randint(2, 8), "chi": rng.choice([32, 64]),
            "cutoff": 1e-6}


# --------------------------------------------------------------------------
# inputs


def _circuit_input(case, seed):
    if case["ops"]:
        return W.nonlocal_ops(case["n"], case["ops"], seed)
    return W.brickwork_u2_su4(case["n"], case["depth"], seed)


def _all_bits(n):
    x = np.arange(1 << n)
    return ((x[:, None] >> np.arange(n - 1, -1, -1)[None, :]) & 1).astype(np.uint8)


def _two_site_input(case, seed):
    a, b = W.random_sites(case["l"], case["m"], case["r"], seed)
    return a.astype(np.complex64), b.astype(np.complex64), W.haar_su4(np.random.default_rng([seed, 1]))


def _batch_sizes(case):
    # widths and bond caps of a batch: spread over 16 .. n_max and 16 .. chi_max
    k, out = case["states"], []
    for i in range(k):
        n = 16 + (case["n_max"] - 16) * i // max(1, k - 1)
        chis = [c for c in (16, 32, 64) if c <= case["chi_max"]]
        out.append((n, chis[i % len(chis)]))
    return out


def _paulis(n):
    zz = ["".join("Z" if k in (i, i + 1) else "I" for k in range(n)) for i in range(n - 1)]
    return zz + ["".join("X" if k == i else "I" for k in range(n)) for i in range(n)]


def _hea(case, seed):
    n = case["n"]
    circ, ang = W.hea_circuit(n, case["layers"], seed)
    layers = [(l.pairs, l.g4) for l in circ.layers]
    axes = ["YZ" if i % 2 == 0 else "" for i in range(len(layers))]
    theta = [ang[i // 2] if i % 2 == 0 else np.zeros((n, 0)) for i in range(len(layers))]
    return layers, axes, theta, _paulis(n), [1.0] * (n - 1) + [0.5] * n


def prepare(case, seed):
    kind, rng = case["kind"], np.random.default_rng(seed)
    s = {"case": case}
    if kind == "circuit":
        s["circuit"] = _circuit_input(case, seed)
        s["bits"] = _all_bits(case["n"])
    elif kind == "gateset":
        s["circuit"] = W.gateset_circuit(case["n"], case["depth"], seed)
        s["bits"] = W.random_bitstrings(case["n"], case["strings"], seed)
        s["mps"] = T.MPS(case["n"], dtype=T.TNSIM_C128, chi_max=case["chi"])
        zero = np.array([1, 0], np.complex128).reshape(1, 2, 1)
        s["zero"] = [zero] * case["n"]
    elif kind == "two_site":
        a, b, g = _two_site_input(case, seed)
        k = max(case["m"], min(case["chi"], 2 * case["l"], 2 * case["r"]))
        s["a"], s["b"] = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
        s["wa"] = torch.zeros(case["l"] * 2 * k, dtype=torch.complex64, device="cuda")
        s["wb"] = torch.zeros(k * 2 * case["r"], dtype=torch.complex64, device="cuda")
        s["g"] = g
    elif kind == "layer":
        s["mps"] = _saturated(case, rng)
        if case["cfg"]:
            T.tnsim_set_jacobi_config(s["mps"].h, case["cfg"])
        s["layers"] = W.brickwork_su4(case["n"], 2, seed).layers
        s["t"] = 0
    elif kind == "batch":
        stream = torch.cuda.Stream()
        s["stream"], s["mps"], layers, keep = stream, [], [[], []], []
        for n, chi in _batch_sizes(case):
            m = _saturated({"n": n, "chi": chi, "dtype": "c64", "gemm": case["gemm"]}, rng, stream.cuda_stream)
            s["mps"].append(m)
            for t, layer in enumerate(W.brickwork_su4(n, 2, int(rng.integers(1 << 31))).layers):
                g = torch.from_numpy(layer.g4.view(np.float64).copy()).cuda()
                keep.append(g)
                layers[t].append((layer.pairs, g.data_ptr(), 0))
        torch.cuda.synchronize()
        s["gates"] = keep
        s["plans"] = [T.tnsim_plan_create([m.h for m in s["mps"]], row) for row in layers]
        s["graph"] = T.tnsim_graph_create(s["plans"])
        s["owner"] = _Graph(s["graph"], s["plans"], s["mps"])
    elif kind in ("amplitudes", "expect", "sample"):
        s["mps"] = _saturated(case, rng)
        if kind == "amplitudes":
            s["bits"] = W.random_bitstrings(case["n"], case["strings"], seed)
        elif kind == "expect":
            s["paulis"] = _paulis(case["n"])
        else:
            s["u"] = rng.random((case["shots"], case["n"]))
    else:
        s["args"] = _hea(case, seed)
        s["params"] = T.tnsim_params_default(T.TNSIM_C128)
        s["params"].chi_max, s["params"].cutoff = case["chi"], case["cutoff"]
    return s


class _Graph:
    """Gives a batch's graph and plans back when its state goes (before the states)."""

    def __init__(self, graph, plans, states):
        self.graph, self.plans, self.states = graph, plans, states

    def __del__(self):
        T.tnsim_graph_destroy(self.graph)
        for p in self.plans:
            T.tnsim_plan_destroy(p)


# --------------------------------------------------------------------------
# one pass


def _real(x, single):
    return x.astype(np.float32) if single else x


def _amps(z, single):
    return z.astype(np.complex64) if single else z


def _spectra(m, bonds, single):
    return _real(np.concatenate([m.spectrum(int(b)) for b in bonds]), single)


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "circuit":
        single = case["dtype"] == "c64"
        m = T.MPS(case["n"], dtype=T.TNSIM_C64 if single else T.TNSIM_C128, chi_max=case["chi"],
                  form=_FORM[case["form"]])
        if case["ops"]:
            m.apply_circuit(s["circuit"])
        else:
            m.run(s["circuit"])
        z = m.amplitudes(s["bits"])
        m.close()
        return _amps(z, single)
    if kind == "gateset":
        m = s["mps"]
        m.import_sites(s["zero"])
        m.run(s["circuit"])
        return m.amplitudes(s["bits"])
    if kind == "two_site":
        a, b, l, r = s["a"], s["b"], case["l"], case["r"]
        s["wa"][:a.numel()].copy_(a.view(-1))
        s["wb"][:b.numel()].copy_(b.view(-1))
        k, eps, sv = T.tnsim_two_site_update_noalloc(s["wa"].data_ptr(), s["wa"].numel(), s["wb"].data_ptr(),
                                                     s["wb"].numel(), l, case["m"], r, s["g"], case["chi"],
                                                     stream=torch.cuda.current_stream().cuda_stream)
        block = s["wa"][:l * 2 * k].view(l * 2, k) @ s["wb"][:k * 2 * r].view(k, 2 * r)
        return {"k": k, "eps": np.float32(eps), "s": _real(sv, True), "block": block}
    if kind == "layer":
        single = case["dtype"] == "c64"
        layer = s["layers"][s["t"] % 2]
        s["t"] += 1
        eps = s["mps"].apply_layer(layer)
        return {"eps": _real(eps, single), "dims": s["mps"].bond_dims(),
                "s": _spectra(s["mps"], layer.pairs + 1, single)}
    if kind == "batch":
        T.tnsim_graph_launch(s["graph"])
        out = {"dims": [], "s": []}
        for m in s["mps"]:
            m.sync()
            out["dims"].append(m.bond_dims())
            out["s"].append(m.spectrum(m.n // 2))
        return {"dims": np.concatenate(out["dims"]), "s": _real(np.concatenate(out["s"]), True)}
    if kind == "amplitudes":
        return _amps(s["mps"].amplitudes(s["bits"]), case["dtype"] == "c64")
    if kind == "expect":
        return _amps(s["mps"].expect_pauli(s["paulis"]), case["dtype"] == "c64")
    if kind == "sample":
        return T.tnsim_sample(s["mps"].h, s["u"])[0]
    layers, axes, theta, paulis, coeffs = s["args"]
    e, g = T.tnsim_grad(case["n"], layers, axes, theta, paulis, coeffs, T.TNSIM_C128, s["params"])
    return {"energy": e, "grad": np.concatenate([x.reshape(-1) for x in g])}


# --------------------------------------------------------------------------
# what a pass cannot do without


def _gate_work(l, m, r, k, es):
    """One two-qubit update: both sites read, both written; the merge, and the least a full
    SVD takes (Golub and Van Loan's count for U, S, V by R-SVD: 4 M^2 N + 22 N^3 with
    M >= N, times 4 for complex arithmetic)."""
    hi, lo = max(2 * l, 2 * r), min(2 * l, 2 * r)
    return (es * 2 * (l * m + m * r + l * k + k * r), 8.0 * 2 * l * m * 2 * r + 4.0 * (4 * hi * hi * lo + 22 * lo ** 3))


def _layer_work(n, chi, parity, es):
    c = _caps(n, chi)
    w = [_gate_work(c[q], c[q + 1], c[q + 2], c[q + 1], es) for q in range(parity, n - 1, 2)]
    return sum(x[0] for x in w), sum(x[1] for x in w)


def work(case):
    kind = case["kind"]
    es = 16 if case.get("dtype", "c64") == "c128" or kind == "grad" else 8
    if kind == "circuit":
        by = fl = 0.0
        for t in range(case["depth"] if not case["ops"] else max(1, case["ops"] // 2)):
            c = _caps(case["n"], min(case["chi"], 1 << min(t + 1, 30)))
            for q in range(t % 2, case["n"] - 1, 2):
                w = _gate_work(c[q], c[q + 1], c[q + 2], c[q + 1], es)
                by, fl = by + w[0], fl + w[1]
        return {"bytes": by + 16 * (1 << case["n"]), "flops": fl + 8.0 * 4 * (1 << case["n"])}
    if kind == "gateset":
        sites = case["n"] * 2 * 4 * 4 * 16
        return {"bytes": case["depth"] * 2 * sites, "flops": case["depth"] * case["n"] / 4 * _gate_work(4, 4, 4, 4, 16)[1]}
    if kind == "two_site":
        w = _gate_work(case["l"], case["m"], case["r"], case["chi"], 8)
        return {"bytes": w[0], "flops": w[1]}
    if kind == "layer":
        w = [_layer_work(case["n"], case["chi"], t, es) for t in (0, 1)]
        return {"bytes": (w[0][0] + w[1][0]) / 2, "flops": (w[0][1] + w[1][1]) / 2}
    if kind == "batch":
        w = [_layer_work(n, chi, t, 8) for n, chi in _batch_sizes(case) for t in (0, 1)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    n = case["n"]
    if kind == "grad":
        # forward, and the adjoint at twice its cost (the usual factor of reverse mode)
        c = _caps(n, min(case["chi"], 1 << min(case["layers"], 30)))
        w = [_gate_work(c[q], c[q + 1], c[q + 2], c[q + 1], es) for q in range(n - 1)]
        return {"bytes": 3.0 * case["layers"] * sum(x[0] for x in w), "flops": 3.0 * case["layers"] * sum(x[1] for x in w)}
    c = _caps(n, case["chi"])
    site = sum(2.0 * c[q] * c[q + 1] for q in range(n)) * es
    env = sum(8.0 * 2 * (c[q] * c[q] * c[q + 1] + c[q] * c[q + 1] * c[q + 1]) for q in range(n))
    if kind == "amplitudes":
        return {"bytes": site + case["strings"] * (n + 16), "flops": case["strings"] * sum(8.0 * c[q] * c[q + 1] for q in range(n))}
    if kind == "expect":
        # left and right environments, and three more transfers per qubit (Z, Z Z and X strings)
        return {"bytes": site + 16 * (2 * n - 1), "flops": 5.0 * env}
    shots = case["shots"]
    per = [min(shots, 1 << min(q, 30)) * (8.0 * c[q] * 2 * c[q + 1] + 8.0 * 2 * c[q + 1] * c[q + 1]) for q in range(n)]
    return {"bytes": site + shots * n * 9, "flops": env + sum(per)}


# --------------------------------------------------------------------------
# the same results in 64 bits, by numpy


def _gated(a, b, g):
    """The gated block of two sites as a matrix, and the sites' outer dimensions."""
    l, r = a.shape[0], b.shape[2]
    m = (a.reshape(2 * l, -1) @ b.reshape(b.shape[0], -1)).reshape(l, 2, 2, r)
    return np.einsum("abcd,lcdr->labr", g.reshape(2, 2, 2, 2), m, optimize=True).reshape(2 * l, 2 * r)


def _kept(sv, chi, cutoff, single, size):
    eps = float(np.finfo(np.float32 if single else np.float64).eps)
    w = sv * sv
    k = max(1, min(chi, int(np.count_nonzero(sv > eps * size * sv[0]))))
    if cutoff > 0.0:
        tail = np.concatenate([np.cumsum(w[::-1])[::-1], [0.0]])
        k = max(1, min(k, int(np.argmax(tail <= cutoff * w.sum()))))
    return k, w[k:].sum() / w.sum(), np.sqrt(w.sum() / w[:k].sum())


def _dense(n, steps):
    """The state vector after steps of (first qubit, second qubit or None, matrix)."""
    psi = np.zeros((2,) * n, np.complex128)
    psi[(0,) * n] = 1.0
    for a, b, g in steps:
        ax = [a] if b is None else [a, b]
        d = len(ax)
        psi = np.tensordot(np.asarray(g).reshape((2,) * (2 * d)), psi, (list(range(d, 2 * d)), ax))
        psi = np.moveaxis(psi, list(range(d)), ax)
    return psi.reshape(-1)


def _steps(circuit):
    for layer in circuit.layers:
        if layer.u1 is not None:
            for q, u in enumerate(layer.u1):
                yield q, None, u
        for q, g in zip(layer.pairs, layer.g4):
            yield int(q), int(q) + 1, g


def _exact_amplitudes(sites, bits):
    v = np.ones((len(bits), 1), np.complex128)
    for q, a in enumerate(sites):
        w = np.empty((len(bits), a.shape[2]), np.complex128)
        for x in (0, 1):
            pick = bits[:, q] == x
            w[pick] = v[pick] @ a[:, x, :]
        v = w
    return v[:, 0]


def _exact_mps(circuit):
    """Sites of the circuit's state without truncation (only zeros are dropped)."""
    n = circuit.n_qubits
    sites = [np.array([1, 0], np.complex128).reshape(1, 2, 1) for _ in range(n)]
    for a, b, g in _steps(circuit):
        if b is None:
            sites[a] = np.einsum("pq,lqr->lpr", g, sites[a])
            continue
        t = _gated(sites[a], sites[b], g)
        u, s, v = np.linalg.svd(t, full_matrices=False)
        k = max(1, int(np.count_nonzero(s > 1e-13 * s[0])))
        sites[a], sites[b] = u[:, :k].reshape(-1, 2, k), (s[:k, None] * v[:k]).reshape(k, 2, -1)
    return sites


def exact(case, seed):
    kind, rng = case["kind"], np.random.default_rng(seed)
    if kind == "circuit":
        c = _circuit_input(case, seed)
        return _dense(case["n"], c if case["ops"] else _steps(c))
    if kind == "gateset":
        return _exact_amplitudes(_exact_mps(W.gateset_circuit(case["n"], case["depth"], seed)),
                                 W.random_bitstrings(case["n"], case["strings"], seed))
    if kind == "two_site":
        a, b, g = _two_site_input(case, seed)
        t = _gated(a.astype(np.complex128), b.astype(np.complex128), g)
        u, sv, v = np.linalg.svd(t, full_matrices=False)
        k, eps, f = _kept(sv, case["chi"], 0.0, True, max(t.shape))
        return {"k": k, "eps": eps, "s": f * sv[:k], "block": (u[:, :k] * (f * sv[:k])) @ v[:k]}
    if kind == "layer":
        single = case["dtype"] == "c64"
        sites = _gauss_sites(case["n"], case["chi"], rng, single)
        layer = W.brickwork_su4(case["n"], 2, seed).layers[0]
        eps, kept, dims = [], [], _caps(case["n"], case["chi"])
        for q, g in zip(layer.pairs, layer.g4):
            t = _gated(sites[q], sites[q + 1], g)
            sv = np.linalg.svd(t, compute_uv=False)
            k, e, f = _kept(sv, case["chi"], case["cutoff"], single, max(t.shape))
            eps.append(e)
            kept.append(f * sv[:k])
            dims[q + 1] = k
        return {"eps": np.array(eps), "dims": np.array(dims, np.int32), "s": np.concatenate(kept)}
    if kind == "amplitudes":
        return _exact_amplitudes(_gauss_sites(case["n"], case["chi"], rng, case["dtype"] == "c64"),
                                 W.random_bitstrings(case["n"], case["strings"], seed))
    if kind == "expect":
        return _exact_terms(_gauss_sites(case["n"], case["chi"], rng, case["dtype"] == "c64"))
    return None


def _exact_terms(sites):
    z, x = np.diag([1.0, -1.0]), np.array([[0.0, 1.0], [1.0, 0.0]])
    n = len(sites)

    def right(a, o, e):   # e: bra index first
        return np.einsum("xpa,pq,ab,yqb->xy", a.conj(), o, e, a, optimize=True)

    R = [None] * n + [np.ones((1, 1), np.complex128)]
    for q in range(n - 1, -1, -1):
        R[q] = right(sites[q], np.eye(2), R[q + 1])
    L = [np.ones((1, 1), np.complex128)]
    for a in sites:
        L.append(np.einsum("xy,xpa,ypb->ab", L[-1], a.conj(), a, optimize=True))
    zz = [np.sum(L[i] * right(sites[i], z, right(sites[i + 1], z, R[i + 2]))) for i in range(n - 1)]
    return np.array(zz + [np.sum(L[i] * right(sites[i], x, R[i + 1])) for i in range(n)])
