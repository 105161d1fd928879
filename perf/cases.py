"""Timed cases of the library: the calls its users make, over the sizes they make them at.

Five kinds of case, each through the public Python binding:

* ``svd``: ``truncated_svd`` of one theta in device memory, the step that a
  two-qubit gate spends most of its time in.  A user goes on to form the
  truncated theta (C V^H) V from it (the product of the two new site
  tensors), so that is what a pass returns, with the kept singular values and
  their count: single vectors are only determined up to a phase, and inside a
  degenerate pair up to a rotation.
* ``theta``: ``contract_theta`` of two complex64 site tensors and a gate.
* ``expect``: ``State.expectations`` of every Jordan-Wigner string of a
  random-integral molecular Hamiltonian on an entangled state.
* ``gates``: ``State.reset``, ``State.apply_gates`` (Haar brickwork from the
  host) and the expectation values of the result.
* ``vqe``: ``vqe_eval`` (one instance, replayed circuit) or
  ``vqe_eval_batch`` (several, one stream each): reset, bind the angles,
  apply the circuit, take the energy.

A case's ``seed`` draws the matrices, tensors, integrals, gates and angles;
sizes and options are in the case.  complex64 paths return float32 values:
that is the precision their results have.
"""

import math
import os

# concurrent evaluations run one stream each: the documented setting for more
# than eight of them, read when CUDA starts
os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")

import numpy as np  # noqa: E402
import torch  # noqa: E402

from paper_2303_03681_gb300 import mps  # noqa: E402
from paper_2303_03681_gb300.inputs import (  # noqa: E402
    brickwork_circuit, hf_bits, jw_molecular_hamiltonian, make_rng, random_integrals, uccsd_template)
from paper_2303_03681_gb300.inputs.circuits import CircuitTemplate  # noqa: E402


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the typical theta of a 50-qubit UCCSD prefix (its median size), with
        # the degenerate pairs that spin symmetry makes
        dict(name="svd_16_pairs", kind="svd", m=16, n=16, precision="fp64", svd_fp64=1, spectrum="pairs"),
        # a ragged theta between unequal bonds, of rank at most chi_m
        dict(name="svd_62x94_deficient", kind="svd", m=62, n=94, precision="fp64", svd_fp64=1,
             spectrum="deficient"),
        # the largest thetas of the 50-qubit workload; ten decades as in the SVD study
        dict(name="svd_124_graded", kind="svd", m=124, n=124, precision="fp64", svd_fp64=1, spectrum="graded"),
        # chi = 256: the large end of the fragment batch
        dict(name="svd_512_graded", kind="svd", m=512, n=512, precision="fp64", svd_fp64=1, spectrum="graded"),
        # complex64 with the FP32 Jacobi SVD: the server's default configuration
        dict(name="svd_c64_200x152", kind="svd", m=200, n=152, precision="fp32", svd_fp64=0, spectrum="graded"),
        # the theta contraction at chi = 512 on the tensor cores
        dict(name="theta_tf32x3_512", kind="theta", chi_l=512, chi_m=512, chi_r=512, precision="tf32x3"),
        # an ordinary ragged theta on the CUDA cores: launch and latency
        dict(name="theta_fp32_45x61x37", kind="theta", chi_l=45, chi_m=61, chi_r=37, precision="fp32"),
        # all 14,251 strings of 10 orbitals on a chi = 64 state
        dict(name="expect_20q_chi64", kind="expect", n=20, layers=6, chi=64, precision="fp64"),
        # 12-qubit brickwork, gates from the host, complex128
        dict(name="gates_12q_8layers", kind="gates", n=12, layers=8, chi=64, precision="fp64"),
        # one 28-qubit UCCSD instance: a long run of small and ordinary gates
        dict(name="vqe_uccsd_28q", kind="vqe", circuit="uccsd", n=28, electrons=10, excitations=20, chi=128,
             precision="fp64", trunc_rel=1e-5, instances=1, chi_typical=24),
        # sixteen fragments at once, the fragment-level parallelism
        dict(name="vqe_uccsd_16q_x16", kind="vqe", circuit="uccsd", n=16, electrons=8, excitations=20, chi=128,
             precision="fp64", trunc_rel=1e-5, instances=16, chi_typical=24),
        # the mixed-precision batched form that the serving line is measured on
        dict(name="vqe_brickwork_12q_tf32x3_x8", kind="vqe", circuit="brickwork", n=12, layers=8, chi=64,
             precision="tf32x3", trunc_rel=1e-5, instances=8),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _even(x):
    return max(4, 2 * int(round(x / 2)))


def draw(rng):
    kind = rng.choice(["svd", "svd", "svd", "theta", "expect", "gates", "vqe", "vqe"])
    if kind == "svd":
        m = _even(_log(rng, 4, 440))
        n = min(440, _even(m * _log(rng, 0.5, 2.0)))
        precision, svd_fp64 = rng.choice([("fp64", 1), ("fp64", 1), ("fp64", 1), ("fp32", 1), ("fp32", 0)])
        return dict(kind=kind, m=m, n=n, precision=precision, svd_fp64=svd_fp64,
                    spectrum=rng.choice(["graded", "pairs", "deficient"]))
    if kind == "theta":
        precision = rng.choice(["fp32", "tf32x3", "bf16x3"])
        a = _log(rng, 4, 128 if precision == "fp32" else 480)
        return dict(kind=kind, chi_l=max(1, int(a * _log(rng, 0.6, 1.0))), chi_m=max(1, int(a * _log(rng, 0.6, 1.0))),
                    chi_r=max(1, int(a * _log(rng, 0.6, 1.0))), precision=precision)
    if kind == "expect":
        layers = rng.randint(3, 6)
        return dict(kind=kind, n=2 * rng.randint(4, 9), layers=layers, chi=2 ** layers,
                    precision=rng.choice(["fp64", "fp64", "fp32"]))
    if kind == "gates":
        return dict(kind=kind, n=rng.randint(4, 12) // 2 * 2, layers=rng.randint(3, 8), chi=64,
                    precision=rng.choice(["fp64", "fp64", "fp32"]))
    n = 2 * rng.randint(4, 9)
    if rng.random() < 0.3:
        return dict(kind="vqe", circuit="brickwork", n=min(n, 12), layers=rng.randint(4, 7), chi=64,
                    precision=rng.choice(["fp32", "tf32x3"]), trunc_rel=1e-5, instances=rng.randint(1, 8))
    return dict(kind="vqe", circuit="uccsd", n=n, electrons=n // 2 // 2 * 2, excitations=rng.randint(6, 20), chi=128,
                precision="fp64", trunc_rel=1e-5, instances=rng.choice([1, 2, 4, 8, 16]), chi_typical=16)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _unitary(rng, n, r):
    q, t = np.linalg.qr(rng.normal(size=(n, r)) + 1j * rng.normal(size=(n, r)))
    return q * (np.diag(t) / np.abs(np.diag(t)))


def _theta_matrix(case, seed):
    """A theta with a prescribed spectrum, unit Frobenius norm, in the storage precision."""
    m, n = case["m"], case["n"]
    rng = make_rng(seed)
    r = min(m, n)
    if case["spectrum"] == "graded":  # ten decades
        s = 10.0 ** -np.linspace(0, 10, r)
    elif case["spectrum"] == "pairs":  # exactly degenerate pairs over six decades
        s = np.repeat(10.0 ** -np.linspace(0, 6, (r + 1) // 2), 2)[:r]
    else:  # half the rank
        s = np.zeros(r)
        s[: r // 2] = np.linspace(1.0, 0.05, r // 2)
    a = (_unitary(rng, m, r) * s) @ _unitary(rng, n, r).conj().T
    a /= np.linalg.norm(a)
    return np.ascontiguousarray(a.astype(np.complex128 if case["precision"] == "fp64" else np.complex64))


def _svd_rule(case):
    """chi_max (even: no cut inside a pair) and the relative threshold: the FP32
    SVD's own rounding of zeros is 1e-7, so it truncates above that."""
    chi_max = max(2, min(case["m"], case["n"]) // 4 * 2)
    return chi_max, (1e-8 if case["precision"] == "fp64" else 1e-7 if case["svd_fp64"] else 1e-5)


def _site_tensors(case, seed):
    rng = make_rng(seed)
    cl, cm, cr = case["chi_l"], case["chi_m"], case["chi_r"]
    s = math.sqrt(2.0 * cm)

    def c64(*shape):
        return ((rng.standard_normal(shape, dtype=np.float32) + 1j * rng.standard_normal(shape, dtype=np.float32))
                / s).astype(np.complex64)

    bl, br = c64(cl, 2, cm), c64(cm, 2, cr)
    return bl, br, _unitary(rng, 4, 4)


def _molecule(case, seed):
    h, g = random_integrals(case["n"] // 2, make_rng(seed))
    return jw_molecular_hamiltonian(h, g)


def _electrons(case):
    return case.get("electrons", case["n"] // 2)


def _template(case, seed):
    if case["circuit"] == "uccsd":
        return uccsd_template(case["n"], case["electrons"], max_excitations=case["excitations"])
    return CircuitTemplate.from_gates(brickwork_circuit(case["n"], case["layers"], make_rng(seed + 1)))


def _angles(case, tmpl, seed):
    rng = make_rng(seed + 2)
    return [rng.uniform(-0.05, 0.05, tmpl.n_params) for _ in range(case["instances"])]


# ---------------------------------------------------------------------------
# a pass
# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    dev = torch.device("cuda", 0)
    if kind == "svd":
        a = _theta_matrix(case, seed)
        stream = torch.cuda.Stream(device=dev)
        chi_max, trunc = _svd_rule(case)
        c = torch.from_numpy(a).to(dev)
        state = dict(case=case, stream=stream, ctx=mps.Context(0, stream=stream), c=c, chi_max=chi_max, trunc=trunc,
                     s=torch.zeros(min(case["m"], case["n"]), dtype=torch.float64, device=dev),
                     vh=torch.zeros((chi_max, case["n"]), dtype=c.dtype, device=dev))
        torch.cuda.synchronize()
        return state
    if kind == "theta":
        bl, br, gate = _site_tensors(case, seed)
        stream = torch.cuda.Stream(device=dev)
        state = dict(case=case, ctx=mps.Context(0, stream=stream), stream=stream, bl=torch.from_numpy(bl).to(dev),
                     br=torch.from_numpy(br).to(dev), gate=gate,
                     out=torch.zeros((2 * case["chi_l"], 2 * case["chi_r"]), dtype=torch.complex64, device=dev))
        torch.cuda.synchronize()
        return state
    if kind in ("expect", "gates"):
        ham = _molecule(case, seed)
        gates = brickwork_circuit(case["n"], case["layers"], make_rng(seed + 1))
        bits = hf_bits(case["n"], _electrons(case))
        ctx = mps.Context(0)
        st = mps.State(ctx, case["n"], bits, chi_max=case["chi"], precision=case["precision"])
        if kind == "expect":
            st.apply_gates(gates)
        return dict(case=case, ctx=ctx, st=st, bits=bits, gates=gates, ham=mps.Hamiltonian(ctx, ham))
    ham, tmpl = _molecule(case, seed), _template(case, seed)
    bits = hf_bits(case["n"], _electrons(case))
    ctxs = [mps.Context(0) for _ in range(case["instances"])]
    circ, h = mps.Circuit(ctxs[0], tmpl), mps.Hamiltonian(ctxs[0], ham)
    states = [mps.State(c, case["n"], bits, chi_max=case["chi"], precision=case["precision"],
                        trunc_rel=case["trunc_rel"]) for c in ctxs]
    return dict(case=case, ctxs=ctxs,
                requests=[(st, circ, h, th, bits) for st, th in zip(states, _angles(case, tmpl, seed))])


def _values(case, x):
    return x if case["precision"] == "fp64" else np.asarray(x, dtype=np.float32)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "svd":
        k, _, _ = mps.truncated_svd(state["ctx"], case["precision"], case["m"], case["n"], state["c"].data_ptr(),
                                    state["chi_max"], state["trunc"], case["svd_fp64"], state["s"].data_ptr(),
                                    state["vh"].data_ptr())
        with torch.cuda.stream(state["stream"]):
            vh = state["vh"][:k]
            theta_k = (state["c"] @ vh.conj().T) @ vh
            s = state["s"][:k].to(torch.float64 if case["precision"] == "fp64" else torch.float32)
        return {"k": k, "s": s, "theta_k": theta_k}
    if kind == "theta":
        mps.contract_theta(state["ctx"], case["precision"], case["chi_l"], case["chi_m"], case["chi_r"],
                           state["bl"].data_ptr(), state["br"].data_ptr(), state["gate"], state["out"].data_ptr())
        return state["out"]
    if kind == "expect":
        return _values(case, state["st"].expectations(state["ham"]))
    if kind == "gates":
        state["st"].reset(state["bits"])
        state["st"].apply_gates(state["gates"])
        return {"values": _values(case, state["st"].expectations(state["ham"])), "chi": state["st"].bond_dims()}
    reqs = state["requests"]
    energies, status = mps.vqe_eval(state["ctxs"][0], reqs) if len(reqs) == 1 else mps.vqe_eval_batch(reqs)
    return {"energies": _values(case, energies), "status": status}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _svd_flops(m, n):
    """Singular values and right vectors by Golub-Kahan (4 m n^2 + 8 n^3 real), complex."""
    m, n = max(m, n), min(m, n)
    return 4.0 * (4.0 * m * n * n + 8.0 * n ** 3)


def _terms(n_orb):
    """Strings of a random-integral Jordan-Wigner Hamiltonian, about (25 orbitals: 571,876)."""
    return 1.46 * n_orb ** 4


def _bond(case, b):
    return min(case["chi"], 2 ** min(b, case["n"] - b))


def _expect_work(case, size, bond):
    """Every string's value read out; each site's tensor meets each operator prefix once."""
    n, terms = case["n"], _terms(case["n"] // 2)
    flops = sum(16.0 * bond(b) ** 3 * terms / n for b in range(1, n))
    tensors = sum(2.0 * size * bond(b) * bond(b + 1) for b in range(n))
    return tensors + 8.0 * terms, flops


def work(case):
    kind = case["kind"]
    size = 16 if case["precision"] == "fp64" else 8
    if kind == "svd":
        m, n, k = case["m"], case["n"], _svd_rule(case)[0]
        return {"bytes": size * (2.0 * m * n + k * n) + 8.0 * k, "flops": _svd_flops(m, n) + 16.0 * m * n * k}
    if kind == "theta":
        cl, cm, cr = case["chi_l"], case["chi_m"], case["chi_r"]
        return {"bytes": 8.0 * (2 * cl * cm + 2 * cm * cr + 4 * cl * cr), "flops": 32.0 * cl * cm * cr}
    if kind == "expect":
        by, fl = _expect_work(case, size, lambda b: _bond(case, b))
        return {"bytes": by, "flops": fl}
    if kind == "gates" or case["circuit"] == "brickwork":
        gates = [(q, layer) for layer in range(case["layers"]) for q in range(layer % 2, case["n"] - 1, 2)]
        fl = sum(_svd_flops(2 * _bond(case, q), 2 * _bond(case, q + 2)) for q, _ in gates)
        by, fe = _expect_work(case, size, lambda b: _bond(case, b))
        k = case.get("instances", 1)
        return {"bytes": k * (by + 300.0 * len(gates)), "flops": k * (fl + fe)}

    def bond(b):
        return min(case["chi_typical"], _bond(case, b))

    span = case["n"] / 2  # a single excitation: two strings, a ladder down and up each
    gates = case["excitations"] * 2 * 2 * span
    by, fe = _expect_work(case, size, bond)
    return {"bytes": case["instances"] * (by + 300.0 * gates),
            "flops": case["instances"] * (fe + gates * _svd_flops(2 * bond(case["n"] // 2), 2 * bond(case["n"] // 2)))}


# ---------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------

def _statevector(n, bits, gates, dev):
    psi = torch.zeros(2 ** n, dtype=torch.complex128, device=dev)
    psi[int("".join(str(int(b)) for b in bits), 2)] = 1.0
    for q, arity, u in zip(gates.q, gates.arity, gates.u):
        d = 2 ** int(arity)
        g = torch.from_numpy(np.ascontiguousarray(np.asarray(u)[:d, :d])).to(dev)
        v = psi.reshape(2 ** int(q), d, -1)
        psi = torch.einsum("ij,ajb->aib", g, v).reshape(-1)
    return psi


def _string_values(n, ham, psi):
    """<psi|P|psi> of every string: P flips the X and Y bits and signs the Z and Y ones."""
    dev = psi.device
    ops = np.asarray(ham.ops)
    w = 1 << np.arange(n - 1, -1, -1, dtype=np.int64)
    x = ((ops == 1) | (ops == 2)) @ w
    z = ((ops == 2) | (ops == 3)) @ w
    ny = (ops == 2).sum(axis=1)
    i = torch.arange(2 ** n, device=dev)
    parity = torch.zeros(2 ** n, dtype=torch.int64, device=dev)
    for b in range(n):
        parity ^= (i >> b) & 1
    sign = 1.0 - 2.0 * parity.to(torch.float64)
    out = torch.empty(ops.shape[0], dtype=torch.complex128, device=dev)
    for t in range(ops.shape[0]):
        out[t] = torch.vdot(psi[i ^ int(x[t])], sign[i & int(z[t])] * psi)
    phase = torch.from_numpy((1j) ** (ny % 4)).to(dev)  # Y|0> = i|1>, Y|1> = -i|0>
    return (phase * out).real


def exact(case, seed):
    kind = case["kind"]
    dev = torch.device("cuda", 0)
    if kind == "svd":
        a = _theta_matrix(case, seed).astype(np.complex128)
        chi_max, trunc = _svd_rule(case)
        u, s, vh = np.linalg.svd(a, full_matrices=False)
        k = max(1, min(chi_max, int(np.count_nonzero(s > trunc * s[0]))))
        return {"k": k, "s": s[:k], "theta_k": (u[:, :k] * s[:k]) @ vh[:k]}
    if kind == "theta":
        bl, br, gate = (torch.from_numpy(np.ascontiguousarray(x)).to(dev, torch.complex128)
                        for x in _site_tensors(case, seed))
        cl, cm, cr = case["chi_l"], case["chi_m"], case["chi_r"]
        t = (bl.reshape(2 * cl, cm) @ br.reshape(cm, 2 * cr)).reshape(cl, 2, 2, cr)
        return torch.einsum("ijkl,aklb->aijb", gate.reshape(2, 2, 2, 2), t).reshape(2 * cl, 2 * cr)
    if case["n"] > 20:
        return None  # a dense state of every instance would take too long
    ham = _molecule(case, seed)
    bits = hf_bits(case["n"], _electrons(case))
    if kind in ("expect", "gates"):
        gates = brickwork_circuit(case["n"], case["layers"], make_rng(seed + 1))
        v = _string_values(case["n"], ham, _statevector(case["n"], bits, gates, dev))
        return v if kind == "expect" else {"values": v, "chi": None}
    tmpl = _template(case, seed)
    coeffs = torch.from_numpy(np.asarray(ham.coeffs, dtype=np.float64)).to(dev)
    energies, known = [], None
    for th in _angles(case, tmpl, seed):
        if known is None or tmpl.n_params:
            known = coeffs @ _string_values(case["n"], ham, _statevector(case["n"], bits, tmpl.bind(th), dev))
        energies.append(float(known))
    return {"energies": np.array(energies), "status": None}
