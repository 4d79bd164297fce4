"""Continuous-input projections (spike_proj_dense) against the CPU oracle
(GPU).  The kernel's FP32 result must lie within the error bound of its
fixed summation tree (depth d = 16 ceil(K / 512) + 5, see spike_proj.h) of
the oracle's near-exact double value; inputs whose every partial sum is
exact in FP32 (one-hot, 0/1 activations) must match bit for bit."""
import math

import numpy as np
import pytest
import torch

import oracle
from gpu_util import DEV, to_dev
from paper_2606_03026_gb300 import spikeproj as sp
from paper_2606_03026_gb300 import synth

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def tree_bound(K, s, mag, y_ref):
    """|y - y_exact| allowed for one output: gamma(d) |s| sum|W x| + 2u |y|."""
    d = 16 * math.ceil(K / 512) + 5
    g = d * U / (1 - d * U)
    return np.abs(s)[None, :] * g * mag + 2 * U * np.abs(y_ref) + 1e-45


def case(seed, N, K, B, ldw=None, ldx=None):
    rng = synth.rng_for(700 + seed, N, K, B)
    ldw = ldw or (K + 15) // 16 * 16
    ldx = ldx or (K + 3) // 4 * 4
    W = rng.integers(-128, 128, size=(N, ldw)).astype(np.int8)          # padding is random
    x = rng.standard_normal((B, ldx)).astype(np.float32)
    x[:, K:] = np.nan                                                   # must never be read
    s = rng.uniform(-2.0, 2.0, N).astype(np.float32)
    return W, x, s, ldw, ldx


def run(problems, B, call=sp.spike_proj_dense):
    """problems: list of (W, x, s, N, K, ldw, ldx); returns the y arrays."""
    keep, args, ys = [], [], []
    for (W, x, s, N, K, ldw, ldx) in problems:
        Wd, xd, sd = to_dev(W), to_dev(x), to_dev(s)
        y = torch.full((B, N + 3), float("nan"), dtype=torch.float32, device=DEV)
        keep += [Wd, xd, sd]
        ys.append(y)
        args.append((Wd, ldw, sd, xd, ldx, y, N + 3, N, K))
    call(args, B)
    torch.cuda.synchronize()
    out = [y.cpu().numpy() for y in ys]
    for y, (W, x, s, N, K, ldw, ldx) in zip(out, problems):
        assert np.isnan(y[:, N:]).all(), "wrote past N"
    return [y[:, :pr[3]] for y, pr in zip(out, problems)]


def check(y, W, x, s, N, K, ldw, what):
    want, mag = oracle.dense(W, s, N, K, x[:, :K], ldq=ldw)
    err = np.abs(y.astype(np.float64) - want)
    bound = tree_bound(K, s.astype(np.float64), mag, want)
    assert np.all(err <= bound), f"{what}: max excess {np.max(err - bound)}"


@pytest.mark.parametrize("N,K", [(1, 1), (5, 17), (33, 513), (100, 1000), (64, 1536),
                                 (7, 6144), (3, 6161)])
@pytest.mark.parametrize("B", [1, 2, 4])
def test_dense_vs_oracle(N, K, B):
    W, x, s, ldw, ldx = case(N + K, N, K, B, ldw=(K + 15) // 16 * 16 + 16, ldx=(K + 3) // 4 * 4 + 4)
    y, = run([(W, x, s, N, K, ldw, ldx)], B)
    check(y, W, x, s, N, K, ldw, f"N={N} K={K} B={B}")


def test_dense_largest_k():
    """K = SPIKE_PROJ_MAX_K (the tree is 16 * 256 + 5 deep) within its bound,
    and an exact case: constant weights and activations 1/4 (every partial
    sum a small dyadic multiple, exact in FP32)."""
    N, K, B = 9, sp.SPIKE_PROJ_MAX_K, 2
    W, x, s, ldw, ldx = case(77, N, K, B)
    y, = run([(W, x, s, N, K, ldw, ldx)], B)
    check(y, W, x, s, N, K, ldw, "K max")
    W = np.full((N, ldw), -3, np.int8)
    x = np.full((B, ldx), 0.25, np.float32)
    y, = run([(W, x, s, N, K, ldw, ldx)], B)
    assert np.array_equal(y, np.broadcast_to(s * np.float32(-0.75 * K), (B, N)))


def test_dense_group_mixed_shapes():
    """Many problems of different shapes in one launch (unit boundaries
    inside and across problems)."""
    shapes = [(1, 1), (4, 32), (5, 100), (9, 1536), (130, 777), (3, 4000), (64, 512), (17, 2049)]
    probs = []
    for i, (N, K) in enumerate(shapes * 3):
        W, x, s, ldw, ldx = case(40 + i, N, K, 3)
        probs.append((W, x, s, N, K, ldw, ldx))
    ys = run(probs, 3)
    for y, (W, x, s, N, K, ldw, ldx) in zip(ys, probs):
        check(y, W, x, s, N, K, ldw, f"group N={N} K={K}")


def test_dense_max_group():
    probs = []
    for i in range(sp.SPIKE_PROJ_DENSE_MAX_GROUP):
        W, x, s, ldw, ldx = case(200 + i, 8 + i % 5, 64 + 32 * (i % 7), 1)
        probs.append((W, x, s, W.shape[0], 64 + 32 * (i % 7), ldw, ldx))
    ys = run(probs, 1)
    for y, (W, x, s, N, K, ldw, ldx) in zip(ys, probs):
        check(y, W, x, s, N, K, ldw, "max group")


def test_dense_exact_cases():
    """One-hot activations give s_m * W[m][k] exactly; 0/1 activations give
    the spike-gated projection's y bit for bit (every partial sum is an
    integer below 2^24); zero activations give zero."""
    N, K, B = 300, 1536, 4
    W, _, s, ldw, ldx = case(9, N, K, B)
    x = np.zeros((B, ldx), np.float32)
    for b, k in enumerate((0, 17, 1023, K - 1)):
        x[b, k] = 1.0
    y, = run([(W, x, s, N, K, ldw, ldx)], B)
    for b, k in enumerate((0, 17, 1023, K - 1)):
        assert np.array_equal(y[b], s * W[:, k].astype(np.float32)), k
    xb = synth.bernoulli(synth.rng_for(710), (B, K), 0.3)
    x = np.zeros((B, ldx), np.float32)
    x[:, :K] = xb
    y, = run([(W, x, s, N, K, ldw, ldx)], B)
    _, ysp = oracle.project(np.ascontiguousarray(W[:, :K].T), s, N, K, xb, "u8")
    assert np.array_equal(y, ysp)
    y, = run([(W, np.zeros((B, ldx), np.float32), s, N, K, ldw, ldx)], B)
    assert not np.any(y)


def test_dense_decode_step_shapes_sampled():
    """The continuous projections of one block at full size (fused QKV 4608,
    attention output 1536, FFN up 6144 rows; K = 1536), one launch, checked
    on sampled rows against the oracle; and run-to-run bit identity."""
    probs = []
    for kind in ("qkv", "out", "up"):
        W, s = synth.dense_weights(0, kind)
        x = synth.hidden_state(0, B=1)
        probs.append((W, x, s, W.shape[0], W.shape[1], W.shape[1], W.shape[1]))
    ys = run(probs, 1)
    again = run(probs, 1)
    rng = synth.rng_for(711)
    for y, y2, (W, x, s, N, K, ldw, ldx) in zip(ys, again, probs):
        assert np.array_equal(y, y2), "not deterministic"
        rows = np.sort(rng.choice(N, 200, replace=False))
        want, mag = oracle.dense(np.ascontiguousarray(W[rows]), s[rows], len(rows), K, x, ldq=ldw)
        err = np.abs(y[:, rows].astype(np.float64) - want)
        assert np.all(err <= tree_bound(K, s[rows].astype(np.float64), mag, want))


# The widest K of the tensor-core form by B, in a problem of many units.
BIG = (4608, 6144)
BIG4 = (9216, 3072)
# A launch takes the tensor-core form where its sizes make that the faster one:
# beside this problem (weights 0) the odd shapes below run there
# (test_host_cpu.py checks it).
FILLER = (600_000, 256)
_filler = {}


def with_filler(args, B):
    """The launch's problems and the filler: (arguments, the filler's y)."""
    N, K = FILLER
    if "W" not in _filler:
        _filler.update(W=torch.zeros(N, K, dtype=torch.int8, device=DEV), s=torch.ones(N, device=DEV))
    x, y = torch.ones(B, K, device=DEV), torch.full((B, N), 3.0, device=DEV)
    return [*args, (_filler["W"], K, _filler["s"], x, K, y, N, N, K)], y


def tensor_form(args, B):
    """One call in the tensor-core form."""
    all_args, y = with_filler(args, B)
    sp.spike_proj_dense(all_args, B)
    assert torch.all(y == 0)


def edge_shapes(B):
    K0 = (BIG if B <= 2 else BIG4)[1]
    return [(1, 1), (15, 15), (16, 16), (17, 17), (33, 63), (7, 64), (31, 65), (48, 511), (16, 512),
            (50, 513), (100, 1000), (16, K0 - 1), BIG if B <= 2 else BIG4, (5, 48), (3, K0)]


@pytest.mark.parametrize("B", [1, 2, 3, 4])
def test_dense_tensor_form_edges(B):
    """The tensor-core form at the edges of its tiles: rows around 16, columns
    around a 16-byte vector, a 64-column chunk and the 8-chunk ring, rows and
    columns of a CTA's share across problems with different activations, two
    problems sharing one activation row, and the widest table."""
    probs = []
    for i, (N, K) in enumerate(edge_shapes(B)):
        big = (N, K) in (BIG, BIG4)
        W, x, s, ldw, ldx = case(300 + i, N, K, B, ldw=None if big else (K + 15) // 16 * 16 + 16)
        probs.append((W, x, s, N, K, ldw, ldx))
    ys = run(probs, B, tensor_form)
    again = run(probs, B, tensor_form)
    rng = synth.rng_for(712, B)
    for y, y2, (W, x, s, N, K, ldw, ldx) in zip(ys, again, probs):
        assert np.array_equal(y, y2), "not deterministic"
        rows = np.arange(N) if N <= 128 else np.sort(rng.choice(N, 128, replace=False))
        check(y[:, rows], np.ascontiguousarray(W[rows]), x, s[rows], len(rows), K, ldw, f"N={N} K={K} B={B}")


@pytest.mark.parametrize("B", [1, 4])
def test_dense_tensor_form_exact_and_shared(B):
    """0/1 activations give the spike-gated projection bit for bit, one-hot
    ones give s_m * W[m][k], with one activation buffer shared by all
    problems of the launch (as a fused query/key/value call has it)."""
    K, N0 = 3072, 8400
    W0, _, s0, ldw, ldx = case(330, N0, K, B)
    xb = synth.bernoulli(synth.rng_for(713), (B, K), 0.3)
    x = np.zeros((B, ldx), np.float32)
    x[:, :K] = xb
    xd, keep, args = to_dev(x), [], []
    for lo, hi in ((0, 8000), (8000, 8017), (8017, N0)):
        y = torch.full((B, hi - lo), float("nan"), device=DEV)
        Wd, sd = to_dev(np.ascontiguousarray(W0[lo:hi])), to_dev(s0[lo:hi])
        keep.append((Wd, sd, y, lo, hi))
        args.append((Wd, ldw, sd, xd, ldx, y, hi - lo, hi - lo, K))
    tensor_form(args, B)
    _, want = oracle.project(np.ascontiguousarray(W0[:, :K].T), s0, N0, K, xb, "u8")
    for _, _, y, lo, hi in keep:
        assert np.array_equal(y.cpu().numpy(), want[:, lo:hi])
    x[:] = 0
    for b in range(B):
        x[b, (17, 0, 1023, K - 1)[b]] = -0.3
    xd.copy_(to_dev(x))
    tensor_form(args, B)
    for _, _, y, lo, hi in keep:
        got = y.cpu().numpy()
        for b in range(B):
            k = (17, 0, 1023, K - 1)[b]
            assert np.array_equal(got[b], s0[lo:hi] * (np.float32(-0.3) * W0[lo:hi, k].astype(np.float32)))


@pytest.mark.parametrize("B", [1, 3])
def test_dense_tensor_form_extreme_activations(B):
    """Activations that three bf16 parts cannot hold (infinite, NaN, subnormal,
    beyond 2^100) are summed with FP32 FMAs, row by row: those rows follow
    IEEE arithmetic and their neighbours are unaffected."""
    vals = [float("inf"), float("-inf"), float("nan"), 1e-40, 3e-38, 1e31, 2.0 ** -100, 2.0 ** 100, 1e-44]
    probs = []
    for i, v in enumerate(vals):
        W, x, s, ldw, ldx = case(350 + i, 40, 200, B)
        x[B - 1, 77] = v
        if abs(v) < 1e-30:
            x[B - 1, :200] = v                     # every activation of the row tiny
        probs.append((W, x, s, 40, 200, ldw, ldx))
        W, x, s, ldw, ldx = case(370 + i, 20, 100, B)
        probs.append((W, x, s, 20, 100, ldw, ldx))
    ys = run(probs, B, tensor_form)
    for y, (W, x, s, N, K, ldw, ldx) in zip(ys, probs):
        with np.errstate(invalid="ignore", over="ignore"):
            want = (x[:, None, :K].astype(np.float64) * W[None, :, :K]).sum(-1) * s
            mag = np.abs(x[:, None, :K].astype(np.float64) * W[None, :, :K]).sum(-1)
        fine = np.isfinite(want)
        assert np.array_equal(np.isnan(want), np.isnan(y))
        assert np.array_equal(want[~fine & ~np.isnan(want)], y[~fine & ~np.isnan(want)])
        # each product and sum near the subnormals may lose 2^-149 once more
        bound = tree_bound(K, s.astype(np.float64), mag, want) + K * 2.0 ** -149
        assert np.all(np.abs(y - want)[fine] <= bound[fine])


def test_dense_errors():
    W = torch.zeros(16, 32, dtype=torch.int8, device=DEV)
    s = torch.ones(16, device=DEV)
    x = torch.ones(1, 32, device=DEV)
    y = torch.zeros(1, 16, device=DEV)
    good = (W, 32, s, x, 32, y, 16, 16, 32)
    bad = [((W, 8, s, x, 32, y, 16, 16, 32), sp.SP_EALIGN),      # ldw < K
           ((W, 32, s, x, 30, y, 16, 16, 32), sp.SP_EALIGN),     # ldx < K
           ((W, 32, s, x, 32, y, 8, 16, 32), sp.SP_EINVAL),      # ldy < N
           ((W, 32, s, x, 32, y, 16, 0, 32), sp.SP_EINVAL),      # N = 0
           ((W, 32, s, x, 32, y, 16, 16, sp.SPIKE_PROJ_MAX_K + 1), sp.SP_ERANGE)]
    for args, status in bad:
        with pytest.raises(sp.SpikeProjError) as e:
            sp.spike_proj_dense([args], 1)
        assert e.value.status == status, args
    with pytest.raises(sp.SpikeProjError):
        sp.spike_proj_dense([good], sp.SPIKE_PROJ_DENSE_MAX_B + 1)
    sp.spike_proj_dense([good], 1)
    torch.cuda.synchronize()
    assert torch.equal(y, torch.zeros_like(y))


def tensor_bound(K, s, mag, want):
    """The bound of the tensor-core form: depth 22 + ceil(K / 64)."""
    d = 22 + (K + 63) // 64
    gamma = d * U / (1 - d * U)
    return np.abs(s) * gamma * mag + U * np.abs(want)


@pytest.mark.parametrize("K", [64, 512, 1536])
@pytest.mark.parametrize("B", [1, 2, 3, 4])
def test_dense_tensor_form_one_large_product(B, K):
    """One product that dwarfs the others of its sum, at every position of a
    64-column chunk, the others of one sign and just below what an FP32 sum of
    its size holds: every addition may lose all of one, which the bound allows
    for.  (A sum of more products than the bound counts on would break it.)"""
    N = 2048
    rng = synth.rng_for(714, K, B)
    W = np.ones((N, K), np.int8)
    W[16:] = rng.integers(1, 128, (N - 16, K))
    s = np.ones(N, np.float32)
    Wd, sd = to_dev(W), to_dev(s)
    rows = np.arange(0, N, 15)
    y = torch.empty(B, N, device=DEV)
    for p0 in range(0, 64, B):
        for small in (1.9921875 * 2.0 ** -25, 1.75 * 2.0 ** -24, 2.0 ** -21):
            x = np.full((B, K), small, np.float32)
            x[:, 1::2] *= np.float32(1 + 2.0 ** -14)          # parts below the leading one too
            for b in range(B):
                x[b, (p0 + b) % 64] = 1.0
            xd = to_dev(x)
            tensor_form([(Wd, K, sd, xd, K, y, N, N, K)], B)
            got = y.cpu().numpy()[:, rows].astype(np.float64)
            prod = x[:, None, :].astype(np.float64) * W[rows][None].astype(np.float64)
            want = prod.sum(-1)
            err = np.abs(got - want)
            worst = (err / tensor_bound(K, 1.0, np.abs(prod).sum(-1), want)).max()
            assert worst <= 1, f"K={K} B={B} position {p0} small {small}: {worst:.2f} of the bound"


@pytest.mark.parametrize("B", [2, 4])
def test_dense_rows_do_not_meet(B):
    """A row's bits depend on its own activations: another row that holds an
    infinity, a NaN or a value that three bf16 parts cannot hold leaves it as
    it is, and the row itself follows IEEE arithmetic."""
    N0, K0 = 4000, 1536
    W, x, s, ldw, ldx = case(400, N0, K0, B)
    W2, x2, s2, ldw2, ldx2 = case(401, 333, 700, B)
    Wd, sd, Wd2, sd2 = to_dev(W), to_dev(s), to_dev(W2), to_dev(s2)

    def call(x, x2):
        y, y2 = torch.full((B, N0), 7.0, device=DEV), torch.full((B, 333), 7.0, device=DEV)
        tensor_form([(Wd, ldw, sd, to_dev(x), ldx, y, N0, N0, K0),
                     (Wd2, ldw2, sd2, to_dev(x2), ldx2, y2, 333, 333, 700)], B)
        return y.cpu().numpy(), y2.cpu().numpy()

    base, base2 = call(x, x2)
    for v in (float("inf"), float("nan"), 1e-40, 1e38):
        for bad in range(B):
            xv, xv2 = x.copy(), x2.copy()
            xv[bad, 77], xv2[bad, 13] = v, v
            got, got2 = call(xv, xv2)
            for b in range(B):
                if b != bad:
                    assert np.array_equal(got[b], base[b]) and np.array_equal(got2[b], base2[b]), (v, bad, b)
            with np.errstate(invalid="ignore", over="ignore"):
                want = (xv2[bad, :700].astype(np.float64) * W2[:, :700]).sum(-1) * s2
            if v != v:
                assert np.isnan(got2[bad]).all()
            elif abs(v) < 1:
                mag = (np.abs(xv2[bad, :700]).astype(np.float64) * np.abs(W2[:, :700])).sum(-1)
                assert np.all(np.abs(got2[bad] - want) <= tree_bound(700, s2.astype(np.float64), mag, want))
