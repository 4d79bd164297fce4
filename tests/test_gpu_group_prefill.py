"""Grouped prefill: the dense tensor-core contraction (ACC = X Q^T, Y = ACC * s
per column; Eq. (sparse) for every row, the 512-token prefill of Section 3.2)
for every member of a group in one persistent launch, through the C ABI,
against the CPU oracle (GPU)."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import DEV, assert_parity, to_dev
from paper_2606_03026_gb300 import spikeproj as sp
from paper_2606_03026_gb300 import synth

pytestmark = pytest.mark.gpu

# ragged members: N not a multiple of the 256-channel tile, K not a multiple
# of the 64-column K block, padded leading dimensions, one-tile members
RAGGED = [(272, 1000, 288), (48, 64, 48), (1536, 777, 1536), (256, 6143, 256),
          (16, 1, 16), (528, 130, 544)]


def make_members(shapes, T, seed=0, p=0.15):
    members = []
    for i, (N, K, ldq) in enumerate(shapes):
        Q, s, x = synth.random_case(700 + seed * 31 + i, N, K, T=T, p=p, ldq=ldq)
        plan = sp.Plan(to_dev(Q), to_dev(s), N, K, ldw=ldq, max_batch=max(T, 1), gemm=True)
        members.append((Q, s, x, N, K, ldq, plan))
    return members


def run_group(group, members, xs_dev, fmt, T, ldx, with_acc=True, with_y=True):
    accs = [torch.full((T, m[3]), -7, dtype=torch.int32, device=DEV) for m in members]
    ys = [torch.full((T, m[3]), -7.0, dtype=torch.float32, device=DEV) for m in members]
    group.prefill(xs_dev, fmt, T, ldx, accs if with_acc else None, ys if with_y else None)
    torch.cuda.synchronize()
    return accs, ys


@pytest.mark.parametrize("T", [1, 129, 200])
@pytest.mark.parametrize("fmt", ["bool8", "u8", "bits"])
def test_ragged_group(T, fmt):
    """Members of different N, K and ldw in one launch, every output against
    the oracle; bool8 rows are read in place, u8 and bit rows staged."""
    members = make_members(RAGGED, T, seed=T)
    group = sp.Group([m[-1] for m in members])
    Kmax = max(m[4] for m in members)
    if fmt == "bits":
        ldx = (Kmax + 31) // 32
        rows = [np.zeros((T, ldx), np.uint32) for _ in members]
        for r, m in zip(rows, members):
            b = synth.pack_bits(m[2])
            r[:, : b.shape[1]] = b
    else:
        ldx = (Kmax + 15) // 16 * 16
        rows = [np.zeros((T, ldx), np.uint8) for _ in members]
        for r, m in zip(rows, members):
            r[:, : m[4]] = m[2] if fmt == "bool8" else m[2] * 3   # u8: any nonzero fires
    xs_dev = [to_dev(r) for r in rows]
    accs, ys = run_group(group, members, xs_dev, fmt, T, ldx)
    for j, (Q, s, x, N, K, ldq, _) in enumerate(members):
        want_acc, want_y = oracle.project(Q, s, N, K, x, "u8", ldq=ldq)
        assert_parity(accs[j], ys[j], want_acc, want_y, f"member {j} ({N}x{K}) {fmt} T={T}")
    assert group.status() == sp.SP_OK
    group.close()


def test_outputs_optional_and_unaligned_rows():
    """acc only, y only, and bool8 rows at an odd byte offset (staged, not
    read in place): same results."""
    T = 131
    members = make_members(RAGGED[:4], T, seed=5)
    group = sp.Group([m[-1] for m in members])
    Kmax = max(m[4] for m in members)
    ldx = (Kmax + 15) // 16 * 16 + 16
    buf = [torch.zeros(T * ldx + 1, dtype=torch.uint8, device=DEV) for _ in members]
    xs_dev = []
    for b, m in zip(buf, members):
        view = b[1:].view(T, ldx)
        view[:, : m[4]] = to_dev(m[2])
        xs_dev.append(view)
    wants = [oracle.project(Q, s, N, K, x, "u8", ldq=ldq) for (Q, s, x, N, K, ldq, _) in members]
    accs, _ = run_group(group, members, xs_dev, "bool8", T, ldx, with_y=False)
    _, ys = run_group(group, members, xs_dev, "bool8", T, ldx, with_acc=False)
    for j, (wa, wy) in enumerate(wants):
        assert_parity(accs[j], ys[j], wa, wy, f"member {j} split outputs")
    group.close()


@pytest.fixture(scope="module")
def prefill22():
    """The 512-token prefill of a 22-block decoder: per block the FFN down
    projection (6144 -> 1536), column rates 0.15 * lognormal(0, 0.5)."""
    blocks = []
    for b in range(22):
        Q, s = synth.prefill_weights(b)
        X = synth.prefill_spikes(b)
        plan = sp.Plan(to_dev(Q), to_dev(s), 1536, 6144, max_batch=512, gemm=True)
        blocks.append((Q, s, X, plan))
    group = sp.Group([b[3] for b in blocks])
    yield blocks, group
    group.close()


def test_prefill_22_blocks(prefill22):
    """22 x (512 x 6144 -> 1536) in one launch, bool8 rows in place: two
    blocks in full and 12 sampled rows of every block against the oracle, and
    every block bit for bit against its own per-plan tensor-core call."""
    blocks, group = prefill22
    T, N, K = 512, 1536, 6144
    xs_dev = [to_dev(X).bool() for (_, _, X, _) in blocks]
    accs = [torch.full((T, N), -7, dtype=torch.int32, device=DEV) for _ in blocks]
    ys = [torch.full((T, N), -7.0, dtype=torch.float32, device=DEV) for _ in blocks]
    group.prefill(xs_dev, "bool8", T, K, accs, ys)
    torch.cuda.synchronize()
    rows = np.array([0, 1, 63, 127, 128, 200, 255, 256, 383, 384, 510, 511])
    for j, (Q, s, X, plan) in enumerate(blocks):
        if j in (0, 21):
            want_acc, want_y = oracle.project(Q, s, N, K, X, "u8")
            assert_parity(accs[j], ys[j], want_acc, want_y, f"block {j} full")
        else:
            want_acc, want_y = oracle.project(Q, s, N, K, X[rows], "u8")
            assert_parity(accs[j][rows], ys[j][rows], want_acc, want_y, f"block {j} rows")
        a1 = torch.empty(T, N, dtype=torch.int32, device=DEV)
        y1 = torch.empty(T, N, dtype=torch.float32, device=DEV)
        plan.batched(xs_dev[j], "bool8", T, K, a1, y1, "gemm")
        torch.cuda.synchronize()
        assert torch.equal(a1, accs[j]), f"block {j}: grouped and per-plan acc differ"
        assert torch.equal(y1.view(torch.int32), ys[j].view(torch.int32)), \
            f"block {j}: grouped and per-plan y differ"
    assert group.status() == sp.SP_OK


def test_prefill_mixed_decoder_group():
    """The 44 binary-input projections of a 22-block decoder (TCAM 1536 ->
    1536 and FFN down 6144 -> 1536 alternating) prefilling 256 tokens in one
    launch: members of different K; sampled rows against the oracle."""
    weights = synth.decode_step_weights(0)
    T = 256
    plans = [sp.Plan(to_dev(Q), to_dev(s), N, K, max_batch=T, gemm=True)
             for (Q, s, N, K) in weights]
    group = sp.Group(plans)
    xs = [synth.prefill_spikes(100 + j, T=T, K=K) for j, (_, _, _, K) in enumerate(weights)]
    ldx = max(w[3] for w in weights)
    rows_np = []
    for x in xs:
        r = np.zeros((T, ldx), np.uint8)
        r[:, : x.shape[1]] = x
        rows_np.append(r)
    xs_dev = [to_dev(r).bool() for r in rows_np]
    accs = [torch.empty(T, w[2], dtype=torch.int32, device=DEV) for w in weights]
    ys = [torch.empty(T, w[2], dtype=torch.float32, device=DEV) for w in weights]
    group.prefill(xs_dev, "bool8", T, ldx, accs, ys)
    torch.cuda.synchronize()
    rows = np.array([0, 5, 127, 128, 255])
    for j, ((Q, s, N, K), x) in enumerate(zip(weights, xs)):
        want_acc, want_y = oracle.project(Q, s, N, K, x[rows], "u8")
        assert_parity(accs[j][rows], ys[j][rows], want_acc, want_y, f"member {j} ({N}x{K})")
    assert group.status() == sp.SP_OK
    group.close()
    for p in plans:
        p.close()


@pytest.mark.parametrize("T,shapes", [
    (256, [(1536, 6144, 1536)] * 3),                  # 2-SM pairs, 18 units split 4 ways
    (100, [(1536, 2000, 1536), (1536, 2048, 1536)]),  # single CTAs, 12 units split 6 ways
    (384, [(1024, 3000, 1024)] * 7 + [(1536, 1536, 1536)] * 9),   # a partial last round
])
def test_tail_split_shapes(T, shapes):
    """Groups whose tiles leave the persistent grid's last round partly idle:
    the tail units run as K ranges on several clusters, each range finishing
    its share of the unit's chunks from all ranges' fp32 partials.  Every
    output against the oracle, twice (the arrival counters are cleared for
    the next launch)."""
    members = make_members(shapes, T, seed=len(shapes))
    group = sp.Group([m[-1] for m in members])
    ldx = max(m[4] for m in members)
    xs_dev = []
    for m in members:
        r = np.zeros((T, ldx), np.uint8)
        r[:, : m[4]] = m[2]
        xs_dev.append(to_dev(r).bool())
    wants = [oracle.project(Q, s, N, K, x, "u8", ldq=ldq) for (Q, s, x, N, K, ldq, _) in members]
    for rep in range(2):
        accs, ys = run_group(group, members, xs_dev, "bool8", T, ldx)
        for j, (wa, wy) in enumerate(wants):
            assert_parity(accs[j], ys[j], wa, wy, f"member {j} rep {rep}")
    assert group.status() == sp.SP_OK
    group.close()


@pytest.mark.parametrize("T,units,K", [
    (256, 30, 640), (256, 24, 1000), (256, 18, 1100), (256, 15, 1280), (256, 5, 1600),   # CTA pairs: 2 to 6 ranges
    (256, 76 + 25, 1030), (250, 12, 520),             # a whole round first; ranges of few K blocks
    (128, 60, 512), (70, 40, 777), (128, 7, 1536),    # single CTAs: 2, 3 and 6 ranges
])
def test_tail_split_ranges(T, units, K):
    """The tail of a grouped launch cut into 2 to 6 K ranges (by the number of
    units of its last round on a 152-SM device), for CTA pairs and single
    CTAs: launches that follow one another without a wait, on alternating
    inputs, all equal to the oracle's rows."""
    shapes, left = [], units
    while left:
        tn = min(left, 11 if left > 22 else 4)
        shapes.append((256 * tn - (16 if left > tn else 112), K, 256 * tn))
        left -= tn
    members = make_members(shapes, T, seed=units)
    group = sp.Group([m[-1] for m in members])
    ldx = (K + 15) // 16 * 16
    inputs = []
    for i in range(2):
        X = [synth.bernoulli(synth.rng_for(7400 + i, units, j), (T, K), 0.2) for j in range(len(members))]
        xs = [torch.zeros(T, ldx, dtype=torch.bool, device=DEV) for _ in members]
        for x, r in zip(X, xs):
            r[:, :K] = to_dev(x).bool()
        rows = np.unique([0, 31, 63, T // 2, T - 1])
        wants = [oracle.project(m[0], m[1], m[3], K, x[rows], "u8", ldq=m[5]) for m, x in zip(members, X)]
        inputs.append((xs, rows, wants))
    outs = []
    for i in range(8):
        accs = [torch.full((T, m[3]), -7, dtype=torch.int32, device=DEV) for m in members]
        ys = [torch.full((T, m[3]), -7.0, dtype=torch.float32, device=DEV) for m in members]
        group.prefill(inputs[i % 2][0], "bool8", T, ldx, accs, ys)
        outs.append((accs, ys))
    torch.cuda.synchronize()
    for i, (accs, ys) in enumerate(outs):
        _, rows, wants = inputs[i % 2]
        for j, (wa, wy) in enumerate(wants):
            assert_parity(accs[j][rows], ys[j][rows], wa, wy, f"launch {i} member {j}")
            if i >= 2:
                assert torch.equal(accs[j], outs[i - 2][0][j]), f"launch {i} member {j} differs from {i - 2}"
    assert group.status() == sp.SP_OK
    group.close()


@pytest.mark.parametrize("T,shapes", [
    (256, [(1536, 700, 1536)] * 5),                   # pairs, 30 units: 2 ranges
    (256, [(1200, 1000, 1216), (1024, 1100, 1024), (1536, 1536, 1536)]),   # pairs, 15 units: 4 ranges
    (256, [(2560, 640, 2560)] * 10),                  # a whole round, then 24 units in 3 ranges
    (130, [(496, 1600, 512)] * 3),                    # pairs with a row tile of two rows
    (100, [(1536, 2000, 1536), (1536, 2048, 1536)]),  # single CTAs, 12 units: 6 ranges
])
def test_tail_ranges_one_after_another(T, shapes):
    """No K range of the tail waits for another one to run: with the whole
    launch on one cluster the ranges of a unit follow each other, every one
    but the last hands all of its chunks over, and the results are exact."""
    members = make_members(shapes, T, seed=len(shapes) + 50)
    group = sp.Group([m[-1] for m in members])
    ldx = (max(m[4] for m in members) + 15) // 16 * 16
    xs_dev = []
    for m in members:
        r = np.zeros((T, ldx), np.uint8)
        r[:, : m[4]] = m[2]
        xs_dev.append(to_dev(r).bool())
    rows = np.unique([0, 31, T // 2, T - 2, T - 1])
    wants = [oracle.project(Q, s, N, K, x[rows], "u8", ldq=ldq) for (Q, s, x, N, K, ldq, _) in members]
    first = None
    for rep in range(4):                              # serial, side by side, serial, side by side
        if rep % 2 == 0:
            group.inject_fault(sp.SP_FAULT_STALL)
        accs, ys = run_group(group, members, xs_dev, "bool8", T, ldx)
        for j, (wa, wy) in enumerate(wants):
            assert_parity(accs[j][rows], ys[j][rows], wa, wy, f"member {j} rep {rep}")
        first = first or accs
        assert all(torch.equal(a, b) for a, b in zip(accs, first)), f"rep {rep}"
        assert group.status() == sp.SP_OK
    group.close()


@pytest.mark.parametrize("fmt", ["u8", "bits", "bool8"])
def test_group_with_a_plan_twice(fmt):
    """A plan that is two members of a group, each with rows of its own: staged
    rows (u8, bits) do not meet in the plan's one staging copy."""
    T, K = 140, 1000
    members = make_members([(272, K, 288), (512, 700, 512)], T, seed=21)
    order = [0, 1, 0, 0]
    group = sp.Group([members[i][-1] for i in order])
    X = [synth.bernoulli(synth.rng_for(7420, j), (T, K), 0.2) for j in range(len(order))]
    if fmt == "bits":
        xs_dev, ldx = [to_dev(synth.pack_bits(x)) for x in X], (K + 31) // 32
    else:
        ldx = 1008
        xs_dev = []
        for x in X:
            r = np.zeros((T, ldx), np.uint8)
            r[:, :K] = x
            xs_dev.append(to_dev(r))
    for rep in range(2):
        accs, ys = run_group(group, [members[i] for i in order], xs_dev, fmt, T, ldx)
        for j, i in enumerate(order):
            Q, s, _, N, Ki, ldq, _ = members[i]
            wa, wy = oracle.project(Q, s, N, Ki, X[j][:, :Ki], "u8", ldq=ldq)
            assert_parity(accs[j], ys[j], wa, wy, f"member {j} rep {rep}")
    assert group.status() == sp.SP_OK
    group.close()


def test_group_prefill_errors():
    members = make_members(RAGGED[:2], 8, seed=9)
    plain = sp.Plan(to_dev(members[0][0]), to_dev(members[0][1]), members[0][3], members[0][4],
                    ldw=members[0][5], max_batch=8)
    xs = [to_dev(np.zeros((8, 1024), np.uint8)) for _ in range(2)]
    out = [torch.empty(8, m[3], dtype=torch.int32, device=DEV) for m in members]
    g_plain = sp.Group([plain, members[1][-1]])
    with pytest.raises(sp.SpikeProjError) as e:
        g_plain.prefill(xs, "bool8", 8, 1024, out, None)
    assert e.value.status == sp.SP_EUNSUPPORTED
    g = sp.Group([m[-1] for m in members])
    with pytest.raises(sp.SpikeProjError) as e:          # T above the plans' max_batch
        g.prefill(xs, "bool8", 9, 1024, out, None)
    assert e.value.status == sp.SP_ERANGE
    with pytest.raises(sp.SpikeProjError) as e:          # neither output
        g.prefill(xs, "bool8", 8, 1024, None, None)
    assert e.value.status == sp.SP_EINVAL
    with pytest.raises(sp.SpikeProjError) as e:          # rows shorter than K
        g.prefill(xs, "bool8", 8, 16, out, None)
    assert e.value.status == sp.SP_EINVAL
    g.close()
    g_plain.close()
