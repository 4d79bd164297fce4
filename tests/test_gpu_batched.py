"""Batched decode and prefill: per-token gather, union shared fetch, the
tcgen05 tensor-core GEMM and the density dispatcher, all against the CPU
oracle and against each other (GPU)."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import DEV, assert_parity, to_dev
from paper_2606_03026_gb300 import spikeproj as sp
from paper_2606_03026_gb300 import synth

pytestmark = pytest.mark.gpu

STRATEGIES = ("gather", "union", "gemm")


def run_batched(plan, spikes, fmt, B, ld, N, strategy):
    acc = torch.full((B, N), -7, dtype=torch.int32, device=DEV)
    y = torch.full((B, N), -7.0, dtype=torch.float32, device=DEV)
    plan.batched(spikes, fmt, B, ld, acc, y, strategy)
    torch.cuda.synchronize()
    return acc, y


@pytest.fixture(scope="module")
def down():
    Qc, s = synth.down_weights(3)
    plan = sp.Plan(to_dev(Qc), to_dev(s), 1536, 6144, max_batch=512, gemm=True)
    return Qc, s, plan


@pytest.mark.parametrize("correlated", [False, True])
@pytest.mark.parametrize("strategy", STRATEGIES + ("auto",))
def test_batch64(down, correlated, strategy):
    """B = 64 tokens, rates U(0.05, 0.2), independent or hot-set correlated."""
    Qc, s, plan = down
    X, _, _ = synth.batched_spikes(0, correlated=correlated)
    want_acc, want_y = oracle.project(Qc, s, 1536, 6144, X, "u8")
    bits = synth.pack_bits(X)
    acc, y = run_batched(plan, to_dev(bits), "bits", 64, bits.shape[1], 1536, strategy)
    assert_parity(acc, y, want_acc, want_y, f"B=64 {strategy} corr={correlated}")
    for fmt in ("u8", "bool8"):
        acc, y = run_batched(plan, to_dev(X), fmt, 64, X.shape[1], 1536, strategy)
        assert_parity(acc, y, want_acc, want_y, f"B=64 {fmt} {strategy} corr={correlated}")
    if strategy == "auto":
        chosen, active = plan.last_dispatch()
        assert chosen in STRATEGIES
        assert active == int(X.astype(np.int64).sum())


def test_prefill_512_tokens(down):
    """512-token prefill block: X ~ Bernoulli(0.15 * lognormal(0, 0.5)); the
    dispatcher must pick the tensor-core GEMM; full output vs the oracle."""
    Qc, s, plan = down
    X = synth.prefill_spikes(0)
    want_acc, want_y = oracle.project(Qc, s, 1536, 6144, X, "u8")
    Xd = to_dev(X)
    acc = torch.empty(512, 1536, dtype=torch.int32, device=DEV)
    y = torch.empty(512, 1536, dtype=torch.float32, device=DEV)
    plan.prefill(Xd, 512, 6144, acc, y, "auto")
    torch.cuda.synchronize()
    assert plan.last_dispatch() == ("gemm", int(X.astype(np.int64).sum()))
    assert_parity(acc, y, want_acc, want_y, "prefill auto")
    for strategy in ("gemm", "gather", "union"):
        acc.fill_(0)
        y.fill_(0)
        plan.prefill(Xd, 512, 6144, acc, y, strategy)
        torch.cuda.synchronize()
        assert_parity(acc, y, want_acc, want_y, f"prefill {strategy}")
    # the same block as 0/1 bytes (a torch.bool tensor): read in place by the GEMM
    Xbool = Xd.bool()
    acc, y = run_batched(plan, Xbool, "bool8", 512, 6144, 1536, "gemm")
    assert_parity(acc, y, want_acc, want_y, "prefill bool8 in place")
    assert plan.status() == sp.SP_OK


@pytest.mark.parametrize("T,N,K,ldq", [(1, 16, 1, 16), (5, 48, 100, 64), (129, 272, 1000, 288),
                                       (300, 1552, 777, 1552), (128, 256, 64, 256),
                                       (257, 512, 6143, 512)])
def test_gemm_ragged(T, N, K, ldq):
    """The tensor-core path on ragged row / column / K-block tails."""
    Qc, s, X = synth.random_case(60 + T, N, K, T=T, p=0.3, ldq=ldq)
    want_acc, want_y = oracle.project(Qc, s, N, K, X, "u8", ldq=ldq)
    plan = sp.Plan(to_dev(Qc), to_dev(s), N, K, ldw=ldq, max_batch=T, gemm=True)
    for strategy in STRATEGIES:
        acc, y = run_batched(plan, to_dev(X), "u8", T, K, N, strategy)
        assert_parity(acc, y, want_acc, want_y, f"T={T} N={N} K={K} {strategy}")


@pytest.mark.parametrize("T,N,K", [(1, 16, 1), (5, 48, 100), (129, 272, 1000), (300, 1552, 777),
                                   (257, 512, 6143)])
def test_gemm_u8_rows_any_nonzero(T, N, K):
    """u8 spike rows on the tensor-core path: any nonzero byte is a spike
    (the 0/1 staging pass maps them), bytes past K in each row are ignored,
    rows and K-blocks ragged."""
    Qc, s, X = synth.random_case(80 + T, N, K, T=T, p=0.3)
    ldx = (K + 15) // 16 * 16 + 16
    rng = synth.rng_for(81, T, K)
    Xs = rng.integers(1, 256, size=(T, ldx)).astype(np.uint8)     # garbage past K
    Xs[:, :K] = np.where(X != 0, rng.integers(1, 256, size=(T, K)), 0).astype(np.uint8)
    want_acc, want_y = oracle.project(Qc, s, N, K, X, "u8")
    plan = sp.Plan(to_dev(Qc), to_dev(s), N, K, max_batch=T, gemm=True)
    for rep in range(2):
        acc, y = run_batched(plan, to_dev(Xs), "u8", T, ldx, N, "gemm")
        assert_parity(acc, y, want_acc, want_y, f"T={T} N={N} K={K} rep {rep}")
    assert plan.status() == sp.SP_OK


@pytest.mark.parametrize("T,N,K", [(1, 16, 1), (5, 48, 100), (129, 272, 1000), (300, 1552, 777),
                                   (257, 512, 6143), (512, 1536, 6144)])
def test_gemm_bool8_rows(T, N, K):
    """0/1 byte rows (SP_SPIKES_BOOL8): with a 16-byte-aligned row stride the
    tensor-core kernel reads them in place (bytes past K ignored, whatever
    they hold); with an odd stride they go through the staging pass.  Both
    equal the oracle and the gather path bit for bit."""
    Qc, s, X = synth.random_case(90 + T, N, K, T=T, p=0.3)
    want_acc, want_y = oracle.project(Qc, s, N, K, X, "u8")
    plan = sp.Plan(to_dev(Qc), to_dev(s), N, K, max_batch=T, gemm=True)
    rng = synth.rng_for(91, T, K)
    for ldx in ((K + 15) // 16 * 16 + 16, K + 1 if (K + 1) % 16 else K + 2):
        Xs = rng.integers(2, 256, size=(T, ldx)).astype(np.uint8)    # not 0/1 past K
        Xs[:, :K] = X != 0
        Xd = to_dev(Xs)
        for strategy in ("gemm", "gemm", "gather"):
            acc, y = run_batched(plan, Xd, "bool8", T, ldx, N, strategy)
            assert_parity(acc, y, want_acc, want_y, f"T={T} N={N} K={K} ldx={ldx} {strategy}")
    assert plan.status() == sp.SP_OK


@pytest.mark.parametrize("T,N,K", [(2, 1536, 6144), (5, 272, 1000), (17, 1552, 777), (33, 1536, 6144),
                                   (64, 528, 3073), (65, 1040, 2049), (3, 2064, 8000), (9, 16, 1)])
def test_gather_rows(T, N, K):
    """The gather strategy on T rows: up to 64 rows run as a group of
    one-row problems (the cluster form when every cluster fits at once, else
    the ticket form with the batched form's workspace offsets; K above 6144
    is always the ticket form), more than 64 in the batched ticket form.
    Rows of mixed rates, every format, twice in a row (the second call must
    find the workspace and tickets clean)."""
    rng = synth.rng_for(95, T, N, K)
    Qc, s, _ = synth.random_case(96 + T, N, K, T=1)
    rates = rng.uniform(0.0, 0.4, size=(T, 1))
    rates[0] = 1.0
    X = (rng.random((T, K)) < rates).astype(np.uint8)
    want_acc, want_y = oracle.project(Qc, s, N, K, X, "u8")
    plan = sp.Plan(to_dev(Qc), to_dev(s), N, K, max_batch=T)
    bits = synth.pack_bits(X)
    for rep in range(2):
        for fmt, rows, ld in (("bits", bits, bits.shape[1]), ("u8", X, K)):
            acc, y = run_batched(plan, to_dev(rows), fmt, T, ld, N, "gather")
            assert_parity(acc, y, want_acc, want_y, f"T={T} N={N} K={K} {fmt} rep {rep}")
    assert plan.status() == sp.SP_OK
    plan.close()


def test_gemm_extremes():
    """All-ones spikes against -128 / +127 weights: the largest sums the
    tensor-core path must carry exactly (|acc| = 128 * K)."""
    T, N, K = 130, 64, 8192
    X = np.ones((T, K), np.uint8)
    X[1::2, ::3] = 0
    s = np.linspace(-2, 2, N).astype(np.float32)
    for c, other in ((-128, 127), (127, -127), (127, 1), (-128, -1)):
        Qc = np.full((K, N), c, np.int8)
        Qc[::5] = other                  # (127, 1) and (-128, -1): large odd sums
        want_acc, want_y = oracle.project(Qc, s, N, K, X, "u8")
        plan = sp.Plan(to_dev(Qc), to_dev(s), N, K, max_batch=T, gemm=True)
        for fmt in ("u8", "bool8"):
            acc, y = run_batched(plan, to_dev(X), fmt, T, K, N, "gemm")
            assert_parity(acc, y, want_acc, want_y, f"gemm extremes {c} {other} {fmt}")


def test_gemm_largest_k():
    """K = SPIKE_PROJ_MAX_K on the tensor-core path: all-ones spikes against
    -128 weights give acc = -2^24 exactly (the exactness boundary), and
    +127 / +1 mixes give large odd sums; K is split 8 ways here."""
    T, N, K = 130, 64, sp.SPIKE_PROJ_MAX_K
    X = np.ones((T, K), np.uint8)
    X[1::2, ::7] = 0
    s = np.linspace(-1, 1, N).astype(np.float32)
    for c, other in ((-128, -128), (127, 1)):
        Qc = np.full((K, N), c, np.int8)
        Qc[::3] = other
        want_acc, want_y = oracle.project(Qc, s, N, K, X, "u8")
        if c == -128:
            assert int(want_acc[0, 0]) == -(1 << 24)
        plan = sp.Plan(to_dev(Qc), to_dev(s), N, K, max_batch=T, gemm=True)
        for fmt in ("bool8", "u8"):
            acc, y = run_batched(plan, to_dev(X), fmt, T, K, N, "gemm")
            assert_parity(acc, y, want_acc, want_y, f"gemm K max {c} {fmt}")
        assert plan.status() == sp.SP_OK
        plan.close()


def test_auto_dispatch_by_cost(down):
    """SP_AUTO: per-token gather for small batches, the tensor-core GEMM for
    large ones on a plan with SP_PLAN_GEMM, never the GEMM without it; the
    result is the same bits either way."""
    Qc, s, plan = down
    X = np.concatenate([synth.batched_spikes(i)[0] for i in range(4)])        # 256 tokens
    want_acc, want_y = oracle.project(Qc, s, 1536, 6144, X, "u8")
    bits = to_dev(synth.pack_bits(X))
    for B, expect in ((8, "gather"), (256, "gemm")):
        acc, y = run_batched(plan, bits, "bits", B, bits.shape[1], 1536, "auto")
        assert plan.last_dispatch()[0] == expect, (B, plan.last_dispatch())
        assert_parity(acc, y, want_acc[:B], want_y[:B], f"auto B={B}")
    plain = sp.Plan(to_dev(Qc), to_dev(s), 1536, 6144, max_batch=256)
    acc, y = run_batched(plain, bits, "bits", 256, bits.shape[1], 1536, "auto")
    assert plain.last_dispatch()[0] == "gather"
    assert_parity(acc, y, want_acc, want_y, "auto without the GEMM operand copy")
    plain.close()


def test_auto_dispatch_second_shape():
    """A 1536 x 1536 projection (the sequence-mixer shape): the small-T
    tensor-core form beats the gather at B = 16, one row and four rows stay
    on the gather (rows run as a group in the cluster form), and every
    choice is exact against the oracle."""
    c = synth.single_projection(4)
    Qc, s = c["Q"], c["s"]
    plan = sp.Plan(to_dev(Qc), to_dev(s), 1536, 1536, max_batch=64, gemm=True)
    rates = np.random.default_rng(5).uniform(0.05, 0.2, size=(64, 1))
    X = (np.random.default_rng(6).random((64, 1536)) < rates).astype(np.uint8)
    want_acc, want_y = oracle.project(Qc, s, 1536, 1536, X, "u8")
    bits = to_dev(synth.pack_bits(X))
    for B, expect in ((1, "gather"), (4, "gather"), (16, "gemm"), (64, "gemm")):
        acc, y = run_batched(plan, bits, "bits", B, bits.shape[1], 1536, "auto")
        assert plan.last_dispatch()[0] == expect, (B, plan.last_dispatch())
        assert_parity(acc, y, want_acc[:B], want_y[:B], f"1536 x 1536 auto B={B}")
    plan.close()


def test_union_many_rows():
    """More rows than one union launch holds (passes of 256)."""
    N, K, B = 256, 2000, 600
    Qc, s, X = synth.random_case(70, N, K, T=B, p=0.05)
    want_acc, want_y = oracle.project(Qc, s, N, K, X, "u8")
    plan = sp.Plan(to_dev(Qc), to_dev(s), N, K, max_batch=B)
    acc, y = run_batched(plan, to_dev(synth.pack_bits(X)), "bits", B, (K + 31) // 32, N, "union")
    assert_parity(acc, y, want_acc, want_y, "union 600 rows")


def test_errors_on_device():
    Qc, s, X = synth.random_case(80, 64, 128, T=4)
    W, S = to_dev(Qc), to_dev(s)
    plan = sp.Plan(W, S, 64, 128, max_batch=4)
    acc = torch.empty(8, 64, dtype=torch.int32, device=DEV)
    with pytest.raises(sp.SpikeProjError) as e:
        plan.batched(to_dev(X), "u8", 5, 128, acc, None, "gather")
    assert e.value.status == sp.SP_ERANGE
    with pytest.raises(sp.SpikeProjError) as e:
        plan.batched(to_dev(X), "u8", 4, 128, acc, None, "gemm")
    assert e.value.status == sp.SP_EUNSUPPORTED
    with pytest.raises(sp.SpikeProjError) as e:
        plan.batched(to_dev(X), "u8", 4, 100, acc, None, "gather")
    assert e.value.status == sp.SP_EINVAL
    with pytest.raises(sp.SpikeProjError) as e:
        plan.decode(to_dev(X[0]), "u8", None, None)
    assert e.value.status == sp.SP_EINVAL
    with pytest.raises(sp.SpikeProjError) as e:
        sp.Plan(W, S, 64, 128, ldw=72)
    assert e.value.status == sp.SP_EALIGN
    assert plan.status() == sp.SP_OK


@pytest.mark.parametrize("fmt", ["u8", "bool8", "bits"])
@pytest.mark.parametrize("shift", [0, 1, 3, 16])
def test_auto_counts_without_waiting(fmt, shift):
    """SP_AUTO where the GEMM is picked whatever the count: the spikes are
    counted by the staging pass (or beside the in-place rows), for rows at any
    alignment and ragged widths, and the count is right when it is asked for
    at once, after several calls in flight, and after an explicit strategy."""
    N, K, T = 1040, 1990, 173
    Qc, s, _ = synth.random_case(91, N, K, T=T)
    plan = sp.Plan(to_dev(Qc), to_dev(s), N, K, ldw=Qc.shape[1], max_batch=T, gemm=True)
    rng = synth.rng_for(7301, shift)
    acc = torch.empty(T, N, dtype=torch.int32, device=DEV)
    y = torch.empty(T, N, dtype=torch.float32, device=DEV)
    for p in (0.15, 0.0, 1.0, 0.4):
        X = synth.bernoulli(rng, (T, K), p)
        if fmt == "bits":
            rows = synth.pack_bits(X)
            buf = to_dev(np.concatenate([np.zeros(shift, rows.dtype), rows.reshape(-1)]).view(np.int32))
            x, ld = buf[shift:], rows.shape[1]
        else:
            ld = 2000 if shift == 16 else K + (3 if shift == 3 else 0)   # 2000: in place for bool8
            pad = np.full((T, ld), 1, np.uint8)                          # past K: never counted
            pad[:, :K] = X * (rng.integers(1, 256, X.shape) if fmt == "u8" else 1)
            buf = to_dev(np.concatenate([np.zeros(shift, np.uint8), pad.reshape(-1)[:(T - 1) * ld + K]]))
            x = buf[shift:]
        for _ in range(3):
            plan.batched(x, fmt, T, ld, acc, y, "auto")
        assert plan.last_dispatch() == ("gemm", int(X.astype(np.int64).sum()))
        want_acc, want_y = oracle.project(Qc, s, N, K, X, "u8", ldq=Qc.shape[1])
        assert_parity(acc, y, want_acc, want_y, f"auto {fmt} shift {shift} p {p}")
        plan.batched(x, fmt, T, ld, acc, y, "gather")
        assert plan.last_dispatch() == ("gemm", int(X.astype(np.int64).sum()))


@pytest.mark.parametrize("N,K", [(1536, 6144), (1536, 1536), (512, 4000), (2064, 3000), (16, 300), (1040, 255),
                                 (48, 12000), (528, 16384)])
def test_batched_gather_cluster_shapes(N, K):
    """The per-token gather over the cluster layouts a batch may take (clusters
    of 16, 12 and 6, one to sixteen chunks, idle tile slots, and the ticket form
    past them): every row equals the single decode and the oracle, at rates
    with one and with several rounds of column loads."""
    Qc, s, _ = synth.random_case(92, N, K)
    plan = sp.Plan(to_dev(Qc), to_dev(s), N, K, ldw=Qc.shape[1], max_batch=64)
    rng = synth.rng_for(7302, N, K)
    for B, p, fmt in ((2, 0.1, "bits"), (3, 1.0, "u8"), (5, 0.3, "bool8"), (8, 0.2, "bits"), (13, 0.5, "bits"),
                      (24, 0.15, "u8"), (40, 0.05, "bits")):
        X = synth.bernoulli(rng, (B, K), p)
        X[B // 2] = 0
        want_acc, want_y = oracle.project(Qc, s, N, K, X, "u8", ldq=Qc.shape[1])
        rows = to_dev(synth.pack_bits(X)) if fmt == "bits" else to_dev(X)
        acc, y = run_batched(plan, rows, fmt, B, rows.shape[1], N, "gather")
        assert_parity(acc, y, want_acc, want_y, f"B={B} p={p} {fmt}")
    assert plan.status() == sp.SP_OK


@pytest.mark.parametrize("N,K", [(512, 600), (512, 130), (1024, 1024), (1536, 1536), (2048, 768), (1040, 1990),
                                 (256, 64), (528, 448), (1536, 3000)])
def test_gemm_split_shapes(N, K):
    """The 128-row GEMM over the K splits it may take (1 to 8 ranges, of 1 to many
    K blocks), at row counts around its tiles."""
    Qc, s, _ = synth.random_case(93, N, K)
    plan = sp.Plan(to_dev(Qc), to_dev(s), N, K, ldw=Qc.shape[1], max_batch=512, gemm=True)
    rng = synth.rng_for(7304, N, K)
    for T in (65, 100, 128, 129, 173, 300, 512):
        X = synth.bernoulli(rng, (T, K), 0.2)
        want_acc, want_y = oracle.project(Qc, s, N, K, X, "u8", ldq=Qc.shape[1])
        rows = to_dev(X)
        acc, y = run_batched(plan, rows, "u8", T, K, N, "gemm")
        assert_parity(acc, y, want_acc, want_y, f"T={T}")
    assert plan.status() == sp.SP_OK


def test_auto_count_is_of_the_call_before():
    """The count read right after an SP_AUTO call that did not wait for it is
    that call's, never the one before (the host may find the sequence number
    of a call in place while it still holds an earlier count, if the two are
    read apart)."""
    N, K, T = 512, 512, 128
    Qc, s, _ = synth.random_case(94, N, K)
    plan = sp.Plan(to_dev(Qc), to_dev(s), N, K, ldw=Qc.shape[1], max_batch=T, gemm=True)
    rng = synth.rng_for(7305)
    X = [synth.bernoulli(rng, (T, K), p) for p in (0.05, 0.6, 0.0, 0.3)]
    want = [("gemm", int(x.astype(np.int64).sum())) for x in X]
    rows = [to_dev(x) for x in X]
    y = torch.empty(T, N, dtype=torch.float32, device=DEV)
    for i in range(4000):
        plan.batched(rows[i % 4], "u8", T, K, None, y, "auto")
        if i % 3:                                # several calls in flight before the question, or none
            assert plan.last_dispatch() == want[i % 4], f"call {i}"
    plan.close()


def test_last_dispatch_beside_a_capture():
    """Asking for a count that is still to come leaves a capture on another
    stream alone."""
    N, K, T = 512, 512, 128
    Qc, s, _ = synth.random_case(95, N, K)
    plan = sp.Plan(to_dev(Qc), to_dev(s), N, K, ldw=Qc.shape[1], max_batch=T, gemm=True)
    X = synth.bernoulli(synth.rng_for(7306), (T, K), 0.2)
    xd = to_dev(X)
    y = torch.empty(T, N, dtype=torch.float32, device=DEV)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    out = torch.ones(8, device=DEV)
    with torch.cuda.stream(a):
        plan.batched(xd, "u8", T, K, None, y, "auto")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(b):
        graph.capture_begin()
        out.add_(1)
    with torch.cuda.stream(a):
        torch.cuda._sleep(20_000_000)                # about 10 ms: the count comes after the question
        plan.batched(xd, "u8", T, K, None, y, "auto")
        assert plan.last_dispatch() == ("gemm", int(X.astype(np.int64).sum()))
    with torch.cuda.stream(b):
        out.mul_(3)
        graph.capture_end()
        graph.replay()
    torch.cuda.synchronize()
    assert torch.all(out == 6)
    plan.close()
