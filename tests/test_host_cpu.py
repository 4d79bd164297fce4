"""The library's host side (launch choice, attributes, error paths) on fake
devices: its objects linked to a stand-in of the CUDA runtime that checks
launches and runs no kernel (fake_cudart.cpp).  No GPU."""
import ctypes
import subprocess
from pathlib import Path

import pytest

from paper_2606_03026_gb300 import _build, spikeproj as sp

HERE = Path(__file__).resolve().parent
FAKE = 1 << 30                                # addresses that no host code reads


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    _build.build()
    out = tmp_path_factory.mktemp("fake") / "libspikeproj_fake.so"
    cuda = Path(_build.nvcc()).resolve().parent.parent / "include"
    objs = [_build.OUT / (src.stem + ".o") for src in _build.sources()]
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-pthread", "-Wl,-Bsymbolic", f"-I{cuda}",
                    f"-I{_build.INCLUDE}", f"-I{_build.CSRC}", str(HERE / "fake_cudart.cpp"), *map(str, objs),
                    "-o", str(out)], check=True)
    lib = ctypes.CDLL(str(out))
    for name, (args, res) in sp._SIGNATURES.items():
        fn = getattr(lib, name)
        fn.argtypes, fn.restype = args, res
    return lib


@pytest.fixture(autouse=True)
def reset(lib):
    lib.fake_fail(b"")
    lib.fake_counts(0, 0)
    lib.fake_device(0)
    lib.fake_launches(), lib.fake_synced()


def make_plan(lib, N=1536, K=6144, rows=512):
    h = ctypes.c_void_p()
    assert lib.spike_proj_plan(ctypes.byref(h), FAKE, N, FAKE, N, K, rows, sp.SP_PLAN_GEMM, None) == sp.SP_OK
    return h


def auto(lib, plan, T=173, K=6144):
    """SP_AUTO on byte rows where the GEMM is picked whatever the count."""
    return lib.spike_proj_batched(plan, FAKE, sp.SP_SPIKES_U8, T, K, FAKE, FAKE, sp.SP_AUTO, None)


def last_dispatch(lib, plan):
    chosen, count = ctypes.c_int(), ctypes.c_int32()
    assert lib.spike_proj_last_dispatch(plan, ctypes.byref(chosen), ctypes.byref(count)) == sp.SP_OK
    return chosen.value, count.value


def dense(lib, shapes, B, own=True):
    """own: every problem has activations of its own."""
    table = (sp.SpDense * len(shapes))()
    for j, (N, K) in enumerate(shapes):
        ld = (K + 15) // 16 * 16
        table[j] = sp.SpDense(FAKE, ld, FAKE, FAKE + own * (j << 20), ld, FAKE, N, N, K)
    return lib.spike_proj_dense(ctypes.addressof(table), len(shapes), B, None)


@pytest.mark.parametrize("first", [0, 1])
def test_every_call_on_either_device(lib, first):
    """What a launch needs of a device (attributes, occupancy, SM count) is
    set on each device a call is made on, not on the first one alone."""
    for dev in (first, 1 - first, first):
        lib.fake_device(dev)
        for B in range(1, sp.SPIKE_PROJ_DENSE_MAX_B + 1):
            assert dense(lib, [(4608, 6144 if B <= 2 else 3072)] * 3, B) == sp.SP_OK, f"dense B={B} on {dev}"
            assert dense(lib, [(64, 256)], B) == sp.SP_OK
        for V, K in ((57344, 1536), (3000, 8192)):
            head = ctypes.c_void_p()
            assert lib.spike_proj_head_create(ctypes.byref(head), FAKE, K, FAKE, V, K, None) == sp.SP_OK
            for B in range(1, 5):
                assert lib.spike_proj_head(head, FAKE, K, B, 0.5, 64, FAKE, None, None, None, None, None, 0,
                                           None) == sp.SP_OK, f"head B={B} K={K} on {dev}"
            assert lib.spike_proj_head_destroy(head) == sp.SP_OK
        plans = [make_plan(lib) for _ in range(2)]
        for T in (1, 5, 16, 64, 100, 512):
            for strategy in ("gather", "gemm", "union"):
                assert lib.spike_proj_batched(plans[0], FAKE, sp.SP_SPIKES_U8, T, 6144, FAKE, FAKE,
                                              sp.KERNELS[strategy], None) == sp.SP_OK, f"{strategy} T={T} on {dev}"
        assert lib.spike_proj_decode(plans[0], FAKE, sp.SP_SPIKES_U8, FAKE, FAKE, None) == sp.SP_OK
        assert lib.spike_proj_lif(FAKE, FAKE, 4096, 8, 4096, 0.9, 1.0, FAKE, 128, None) == sp.SP_OK
        group = ctypes.c_void_p()
        two = (ctypes.c_void_p * 2)(*plans)
        rows = (ctypes.c_void_p * 2)(FAKE, FAKE)
        assert lib.spike_proj_group_create(ctypes.byref(group), two, 2, None) == sp.SP_OK
        assert lib.spike_proj_group_decode(group, FAKE, sp.SP_SPIKES_U8, 6144, FAKE, FAKE, 1536, None) == sp.SP_OK
        for T in (100, 256):                  # single CTAs and CTA pairs
            assert lib.spike_proj_group_prefill(group, rows, sp.SP_SPIKES_BOOL8, T, 6144, rows, rows,
                                                None) == sp.SP_OK, f"group prefill T={T} on {dev}"
        assert lib.spike_proj_group_destroy(group) == sp.SP_OK
        for p in plans:
            assert lib.spike_proj_plan_destroy(p) == sp.SP_OK


def test_count_after_a_failed_launch(lib):
    """A GEMM that cannot be launched after the pass that counts the spikes
    has been: the next call's count is its own."""
    plan = make_plan(lib)
    lib.fake_counts(100, 0)
    lib.fake_fail(b"gemm_kernel")
    for _ in range(2):
        assert auto(lib, plan) == sp.SP_ECUDA
    lib.fake_fail(b"")
    lib.fake_counts(70, 0)
    assert auto(lib, plan) == sp.SP_OK
    assert last_dispatch(lib, plan) == (sp.SP_GEMM, 70)
    assert lib.spike_proj_plan_destroy(plan) == sp.SP_OK


def test_last_dispatch_waits_without_the_device(lib):
    """The count of a call that did not wait for it is waited for on the host:
    no synchronisation, which would stall other streams and break a capture
    elsewhere.  A count that never comes is -1 and not an earlier call's, after
    a synchronisation of the plan's own device."""
    lib.fake_device(1)
    plan = make_plan(lib)
    lib.fake_device(0)
    for active, ms in ((5, 0), (90, 60), (12, 5)):
        lib.fake_counts(active, ms)
        assert auto(lib, plan) == sp.SP_OK
        assert last_dispatch(lib, plan) == (sp.SP_GEMM, active)
        assert lib.fake_synced() == -1
    lib.fake_counts(33, -1)
    assert auto(lib, plan) == sp.SP_OK
    assert last_dispatch(lib, plan) == (sp.SP_GEMM, -1)
    assert lib.fake_synced() == 1
    device = ctypes.c_int()
    assert lib.cudaGetDevice(ctypes.byref(device)) == 0 and device.value == 0
    assert lib.spike_proj_plan_destroy(plan) == sp.SP_OK


def test_last_dispatch_after_a_failed_call(lib):
    """A call that fails leaves the call before it the last one."""
    plan = make_plan(lib)
    lib.fake_counts(41, 30)
    assert auto(lib, plan) == sp.SP_OK
    lib.fake_fail(b"spikes_to_01")
    assert auto(lib, plan) == sp.SP_ECUDA
    assert last_dispatch(lib, plan) == (sp.SP_GEMM, 41)
    assert lib.spike_proj_plan_destroy(plan) == sp.SP_OK


def is_tensor_form(lib, shapes, B, own=True):
    assert dense(lib, shapes, B, own) == sp.SP_OK
    assert lib.fake_last_is(b"dense_kernel") or lib.fake_last_is(b"dense_mma_kernel")
    return bool(lib.fake_last_is(b"dense_mma_kernel"))


def test_dense_form(lib):
    """The form of a continuous-input launch: the tensor cores where they were
    measured to be the faster one or close to it (decode steps, large
    launches), FMAs where those were (small and wide launches, many problems of
    few rows with activations of their own)."""
    step = [(n, 1536) for _ in range(22) for n in (4608, 1536, 6144)]
    for B in (1, 2, 3, 4):
        assert is_tensor_form(lib, step, B) and is_tensor_form(lib, step, B, own=False)
        assert not is_tensor_form(lib, [(64, 1536)], B)
        assert not is_tensor_form(lib, [(4096, 16384)], B)           # K without a table
        assert is_tensor_form(lib, [(200_000, 128)], B)
    for shapes, B in (([(52, 3000)] * 64, 3), ([(136, 3000)] * 64, 3), ([(66, 6144)] * 64, 1), ([(152, 6144)] * 64, 1),
                      ([(65, 6144)] * 64, 2)):
        assert not is_tensor_form(lib, shapes, B), (shapes[0], len(shapes), B)
    for shapes, B in (([(13020, 768)], 2), ([(6000, 3000)], 4), ([(3000, 3000)], 4), ([(11718, 1536)], 3),
                      ([(78125, 768)], 1), ([(65104, 1536)], 2), ([(406, 768)] * 64, 4)):
        assert is_tensor_form(lib, shapes, B), (shapes[0], len(shapes), B)


def test_dense_form_of_the_gpu_tests(lib):
    """The launches that test_gpu_dense.py means for the tensor-core form."""
    import test_gpu_dense as t
    for B in (1, 2, 3, 4):
        assert is_tensor_form(lib, [*t.edge_shapes(B), t.FILLER], B)
        assert is_tensor_form(lib, [(8000, 3072), (17, 3072), (383, 3072), t.FILLER], B, own=False)
        assert is_tensor_form(lib, [s for _ in range(9) for s in ((40, 200), (20, 100))] + [t.FILLER], B)
        assert is_tensor_form(lib, [(4000, 1536), (333, 700), t.FILLER], B)
        for K in (64, 512, 1536):
            assert is_tensor_form(lib, [(2048, K), t.FILLER], B)
