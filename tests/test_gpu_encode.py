"""Amplitude-encoded input (slos_encoded_forward): psi(t) = sum_s <t|U|s> x_s
against the oracle's transfer matrix (Ryser permanents)."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2602_11092_gb300 import workloads

pytestmark = pytest.mark.gpu

P_TOL = 1e-5


def rand_states(rng, B, K):
    x = rng.standard_normal((B, K)) + 1j * rng.standard_normal((B, K))
    return (x / np.linalg.norm(x, axis=1, keepdims=True)).astype(np.complex64)


@pytest.mark.parametrize("m,n,space,B", [(4, 3, 0, 5), (6, 3, 0, 70), (5, 4, 0, 3), (8, 3, 1, 9), (7, 7, 0, 2),
                                         (9, 1, 0, 4)])
def test_encoded_amplitudes_match_oracle(slos, m, n, space, B):
    rng = np.random.default_rng(80 + m + n)
    s = [n] + [0] * (m - 1)  # any input: the plan only fixes (m, n, space)
    if space == 1:
        s = [1] * n + [0] * (m - n)
    plan = slos.Plan(m, s, space=space)
    basis = oracle.enumerate_unbunched(m, n) if space == 1 else oracle.enumerate_fock(m, n)
    K = plan.n_outputs
    assert K == len(basis)
    U = workloads.haar_unitaries(m, 1, rng)[0].astype(np.complex64)
    X = rand_states(rng, B, K)
    Ut, Xt = torch.tensor(U, device="cuda"), torch.tensor(X, device="cuda")
    amps = plan.encoded_forward(Ut, Xt, slos.AMPS).cpu().numpy()
    probs = plan.encoded_forward(Ut, Xt, slos.PROBS).cpu().numpy()
    ref = oracle.encoded_amplitudes(U.astype(np.complex128), X.astype(np.complex128), basis)
    assert np.abs(amps - ref).max() <= P_TOL
    assert np.abs(probs - np.abs(ref) ** 2).max() <= P_TOL
    if space == 0:  # the transfer matrix is unitary on the full Fock basis
        assert np.abs(probs.sum(axis=1) - 1.0).max() <= 1e-4


@pytest.mark.parametrize("m,n,B", [(8, 4, 4100), (10, 4, 130), (12, 2, 9000)])
def test_encoded_tensor_core_gemm_chunks_and_ragged_tiles(slos, m, n, B):
    """The GEMM runs on the tensor cores in TF32 with the three-product split
    (batch chunks of 4096 rows, 128 x 256 output tiles over (re, im)
    interleaved columns): batches past one chunk, output counts that leave a
    partial tile (2K = 660, 1430, 156 columns), every row and output against
    the oracle within the FP32 tolerance."""
    rng = np.random.default_rng(300 + m + n)
    plan = slos.Plan(m, [n] + [0] * (m - 1))
    basis = oracle.enumerate_fock(m, n)
    K = plan.n_outputs
    U = workloads.haar_unitaries(m, 1, rng)[0].astype(np.complex64)
    X = rand_states(rng, B, K)
    Ut, Xt = torch.tensor(U, device="cuda"), torch.tensor(X, device="cuda")
    amps = plan.encoded_forward(Ut, Xt, slos.AMPS)
    probs = plan.encoded_forward(Ut, Xt, slos.PROBS)
    plan.sync_status()
    ref = oracle.encoded_amplitudes(U.astype(np.complex128), X.astype(np.complex128), basis)
    assert np.abs(amps.cpu().numpy() - ref).max() <= P_TOL
    p = probs.cpu().numpy()
    assert np.abs(p - np.abs(ref) ** 2).max() <= P_TOL
    assert 0.5 * np.abs(p - np.abs(ref) ** 2).sum(axis=1).max() <= 1e-5
    assert torch.equal(probs, plan.encoded_forward(Ut, Xt, slos.PROBS))  # fixed summation order


def test_encoded_basis_state_equals_plain_forward(slos):
    """x = |s> reproduces slos_forward's amplitudes for input s."""
    m, s = 10, [1, 0, 2, 0, 1, 0, 0, 0, 0, 0]
    rng = np.random.default_rng(91)
    plan = slos.Plan(m, s)
    U = torch.tensor(workloads.haar_unitaries(m, 1, rng)[0].astype(np.complex64), device="cuda")
    basis = oracle.enumerate_fock(m, 4)
    idx = [i for i, t in enumerate(basis) if list(t) == s][0]
    X = torch.zeros((2, plan.n_outputs), dtype=torch.complex64, device="cuda")
    X[0, idx] = 1.0
    X[1, idx] = 1j
    amps = plan.encoded_forward(U, X, slos.AMPS)
    ref = plan.forward(U[None], slos.AMPS)[0]
    assert (amps[0] - ref).abs().max().item() <= P_TOL
    assert (amps[1] - 1j * ref).abs().max().item() <= P_TOL


def test_encoded_rejects_large_or_threshold_plans(slos):
    with pytest.raises(slos.SlosError):
        slos.Plan(16, [1, 0] * 8).encoded_forward(torch.eye(16, dtype=torch.complex64, device="cuda"),
                                                   torch.zeros((1, 490314), dtype=torch.complex64, device="cuda"))
    with pytest.raises(slos.SlosError):
        slos.Plan(4, [1, 1, 0, 0], slos.THRESHOLD).encoded_forward(
            torch.eye(4, dtype=torch.complex64, device="cuda"), torch.zeros((1, 10), dtype=torch.complex64,
                                                                            device="cuda"))


@pytest.mark.parametrize("m,n,B", [(5, 2, 6), (6, 3, 131), (11, 5, 5), (2, 7, 1)])
def test_encoded_rows_and_outputs_of_any_scale(slos, m, n, B):
    """The operands are split into FP16 pairs at a scale of their own per
    state vector and per output: vectors of norms 1e-20 to 1e15 and a zero
    vector, and a lossy map (one mode damped by 1e-5, so outputs with many
    photons there are 1e-25 of the others), odd output counts and ones beyond
    a row's registers.  Every vector and every output keeps the relative
    accuracy of its own size: the split's 2^-22 and the FP32 recursion's few
    ulps, accumulated over the sum, against an FP64 restatement."""
    rng = np.random.default_rng(17 * m + n)
    plan = slos.Plan(m, [n] + [0] * (m - 1))
    basis = oracle.enumerate_fock(m, n)
    K = plan.n_outputs
    U = workloads.haar_unitaries(m, 1, rng)[0]
    U[1, :] *= 1e-5
    U = U.astype(np.complex64)
    X = rand_states(rng, B, K).astype(np.complex128)
    X *= (10.0 ** rng.uniform(-20, 15, size=B))[:, None]
    X[B // 2] = 0.0
    X = X.astype(np.complex64)
    amps = plan.encoded_forward(torch.tensor(U, device="cuda"), torch.tensor(X, device="cuda"), slos.AMPS).cpu().numpy()
    ref = oracle.encoded_amplitudes(U.astype(np.complex128), X.astype(np.complex128), basis)
    norm = np.linalg.norm(X.astype(np.complex128), axis=1)
    size = np.abs(oracle.transfer_matrix(U.astype(np.complex128), basis)).max(axis=1)  # largest entry of each output
    bound = 4e-6 * np.sqrt(K) * norm[:, None] * size[None, :]
    assert np.all(np.abs(amps - ref) <= bound + 1e-44)
    assert np.all(amps[B // 2] == 0)


@pytest.mark.parametrize("m,n,B", [(3, 1, 1), (6, 3, 130), (7, 3, 257), (8, 4, 513), (9, 4, 40), (10, 4, 300), (9, 5, 1100)])
@pytest.mark.parametrize("kind", ["amps", "probs"])
def test_encoded_tile_widths(slos, m, n, B, kind):
    """Output counts and batches whose tiles take widths from 32 to 256
    columns, ragged in both directions and odd row lengths, against the FP64
    product with the transfer matrix."""
    rng = np.random.default_rng(m * 100 + B)
    plan = slos.Plan(m, [n] + [0] * (m - 1))
    basis = oracle.enumerate_fock(m, n)
    U = workloads.haar_unitaries(m, 1, rng)[0].astype(np.complex64)
    X = rand_states(rng, B, plan.n_outputs).astype(np.complex64)
    out = slos.AMPS if kind == "amps" else slos.PROBS
    got = plan.encoded_forward(torch.tensor(U, device="cuda"), torch.tensor(X, device="cuda"), out).cpu().numpy()
    ref = X.astype(np.complex128) @ oracle.transfer_matrix(U.astype(np.complex128), basis).T
    # the split's 2^-22 and the FP32 recursion and sums, on amplitudes of norm 1
    if kind == "amps":
        assert np.abs(got - ref).max() <= 4e-6
    else:
        assert np.abs(got - np.abs(ref) ** 2).max() <= 8e-6


def transfer_by_recursion(U, m, n):
    """Phi in FP64 by the photon-by-photon recursion: products and sums of
    entries of U only, so zeros and small entries are exact to their own size
    (a permanent by inclusion and exclusion leaves 1e-17 in their place)."""
    layers = [oracle.enumerate_fock(m, k) for k in range(n + 1)]
    rank = [{tuple(int(x) for x in t): i for i, t in enumerate(b)} for b in layers]
    A = {(0,) * m: np.ones(1, dtype=np.complex128)}
    for k in range(1, n + 1):
        child = np.array([[rank[k][tuple(int(x) + (q == j) for q, x in enumerate(t))] for j in range(m)]
                          for t in layers[k - 1]])
        cur = {}
        for s in rank[k]:
            c = max(q for q in range(m) if s[q])
            prev = A[tuple(x - (q == c) for q, x in enumerate(s))]
            v = np.zeros(len(layers[k]), dtype=np.complex128)
            for j in range(m):
                v[child[:, j]] += U[j, c] * prev
            cur[s] = v
        A = cur
    g = np.sqrt([np.prod([math.factorial(int(x)) for x in t]) for t in layers[n]])
    return np.stack([A[s] for s in rank[n]], axis=1) * g[:, None] / g[None, :]


@pytest.mark.parametrize("m,n,B", [(6, 3, 131), (9, 4, 40), (10, 4, 300)])
@pytest.mark.parametrize("u", ["phases", "permutation", "positive"])
def test_encoded_components_of_very_different_size(slos, u, m, n, B):
    """State vectors whose components span 25 orders of magnitude through maps
    that do not mix (phases, a permutation): every output has one term and
    keeps that component's relative accuracy, however small it is beside the
    rest of its vector.  `positive`: a map with entries from 1e-8 to 1, all
    sums of positive terms, so every output is as accurate as its terms.
    Per term: the operands' 24 bits, about 2 n + 4 FP32 roundings of the
    recursion and the factorials, the sums' truncation over 24 MMAs (below
    2^-20): 4e-6 of the output's own size."""
    rng = np.random.default_rng(10 * m + n)
    plan = slos.Plan(m, [n] + [0] * (m - 1))
    K = plan.n_outputs
    span = 10.0 ** rng.uniform(-25, 0, (B, K))
    if u == "positive":
        U = (10.0 ** rng.uniform(-8, 0, (m, m))).astype(np.complex64)
        X = span.astype(np.complex64)
        X[: B // 2] *= np.arange(K)[None, :] == rng.integers(0, K, B // 2)[:, None]  # basis states: entries of Phi
    else:
        U = np.diag(np.exp(2j * np.pi * rng.random(m)))
        if u == "permutation":
            U = U[rng.permutation(m)]
        U = U.astype(np.complex64)
        X = (span * np.exp(2j * np.pi * rng.random((B, K)))).astype(np.complex64)
    got = plan.encoded_forward(torch.tensor(U, device="cuda"), torch.tensor(X, device="cuda"), slos.AMPS).cpu().numpy()
    ref = X.astype(np.complex128) @ transfer_by_recursion(U.astype(np.complex128), m, n).T
    assert np.all(np.abs(got - ref) <= 4e-6 * np.abs(ref) + 1e-37)


@pytest.mark.parametrize("m,n,B", [(2, 1, 1), (3, 1, 130), (4, 2, 5000), (2, 11, 20), (4, 4, 77), (10, 2, 12), (6, 3, 3001),
                                   (16, 1, 17), (3, 9, 9), (11, 2, 40), (22, 1, 700)])
@pytest.mark.parametrize("kind", ["amps", "probs"])
def test_encoded_small_bases(slos, m, n, B, kind):
    """Bases of 2 to 66 states (both sides of the FP32 product's 64): vectors
    that do not fill the last CTA, more of them than the grid takes at once.
    FP32 recursion, products and sums of at most 66 terms."""
    rng = np.random.default_rng(31 * m + B)
    plan = slos.Plan(m, [n] + [0] * (m - 1))
    U = workloads.haar_unitaries(m, 1, rng)[0].astype(np.complex64)
    X = rand_states(rng, B, plan.n_outputs).astype(np.complex64)
    out = slos.AMPS if kind == "amps" else slos.PROBS
    got = plan.encoded_forward(torch.tensor(U, device="cuda"), torch.tensor(X, device="cuda"), out)
    assert torch.equal(got, plan.encoded_forward(torch.tensor(U, device="cuda"), torch.tensor(X, device="cuda"), out))
    got = got.cpu().numpy()
    ref = X.astype(np.complex128) @ transfer_by_recursion(U.astype(np.complex128), m, n).T
    if kind == "amps":
        assert np.abs(got - ref).max() <= 4e-6
    else:
        assert np.abs(got - np.abs(ref) ** 2).max() <= 8e-6
