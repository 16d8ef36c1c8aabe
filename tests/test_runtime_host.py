"""Host code of the library on a CUDA runtime that only keeps count (fake_cudart)."""
import ctypes

import pytest

import paper_2105_07298_gb300 as apsp
from fake_cudart import load, word

DEV = ctypes.c_void_p(256)  # stands for any device buffer: nothing reads it


@pytest.fixture()
def lib(tmp_path):
    return load(tmp_path)


def _one_shot(lib):
    n, off = (ctypes.c_int32 * 2)(8, 16), (ctypes.c_int64 * 2)(0, 64)
    return lib.apsp_fw_batched_f32(DEV, DEV, n, off, 2, None)


def test_one_shot_batch_refuses_graph_capture(lib):
    """Its work list is uploaded from memory of the call, which a replay would not find."""
    word(lib, "capturing").value = 1
    assert _one_shot(lib) == apsp.APSP_ECUDA
    assert not any(word(lib, w).value for w in ("launches", "copies", "allocs", "pool_allocs", "live"))
    word(lib, "capturing").value = 0
    assert _one_shot(lib) == apsp.APSP_OK
    assert word(lib, "launches").value == word(lib, "copies").value == 1 and word(lib, "live").value == 0


def test_device_status_reads_and_clears_every_error_word(lib):
    """Each source file's kernels have a word of their own."""
    words = [lib.var_at(i) for i in range(word(lib, "num_vars").value) if b"g_device_error" in lib.var_name(i)]
    assert len(words) >= 5 and lib.apsp_device_status(None) == apsp.APSP_OK
    for w in words:
        ctypes.c_int.from_address(w).value = apsp.APSP_ETIMEOUT
        assert lib.apsp_device_status(None) == apsp.APSP_ETIMEOUT
        assert lib.apsp_device_status(None) == apsp.APSP_OK


def _counts(lib, *names):
    return tuple(word(lib, w).value for w in names)


@pytest.mark.parametrize("error", [2, 1])  # out of memory, and any other
def test_scratch_falls_back_to_the_default_pool(lib, error):
    word(lib, "pool_error").value = error
    for call in (1, 2):
        assert _one_shot(lib) == apsp.APSP_OK
        assert _counts(lib, "pools_created", "pools_destroyed", "pool_allocs", "pools_trimmed", "allocs",
                       "live") == (1, 0, call, call, call, 0)
    word(lib, "alloc_error").value = 2
    assert _one_shot(lib) == apsp.APSP_ENOMEM
    word(lib, "pool_error").value = word(lib, "alloc_error").value = 0
    assert _one_shot(lib) == apsp.APSP_OK
    assert _counts(lib, "pools_created", "allocs", "live") == (1, 3, 0)


def test_scratch_pool_without_its_bound_is_not_kept(lib):
    """The bound on what it keeps could not be set: the default pool serves."""
    word(lib, "pool_attr_error").value = 1
    assert _one_shot(lib) == apsp.APSP_OK
    assert _counts(lib, "pools_created", "pools_destroyed", "pool_allocs", "allocs") == (1, 1, 0, 1)


@pytest.mark.parametrize("fn,n", [("apsp_fw_f32", 2900), ("apsp_fw_f64", 4000), ("apsp_fw_f32", 1000)])
def test_phase_timing_counts_every_launch(lib, fn, n):
    """Also the dense kernel behind each screen."""
    lib.apsp_profile_enable(1)
    assert getattr(lib, fn)(DEV, ctypes.c_int64(n), ctypes.c_int64(n), DEV, None) == apsp.APSP_OK
    ms, launches = (ctypes.c_double * 4)(), (ctypes.c_int64 * 4)()
    assert lib.apsp_profile_collect(ms, launches) == apsp.APSP_OK
    assert sum(launches) == word(lib, "launches").value
    R = (n + 127) // 128
    assert launches[:3] == [1, R, R] and (launches[3] == 2 * R - 1) == (n == 1000)
    lib.apsp_profile_enable(0)


@pytest.mark.parametrize("fn,n", [("apsp_fw_f32", 1000), ("apsp_fw_f32", 2900), ("apsp_fw_f64", 4000)])
def test_no_launch_starts_before_its_predecessor_ends(lib, fn, n):
    """Its waiting CTAs could hold the SMs that another stream's kernel, which they come to wait
    for in a shared hardware queue, needs."""
    assert getattr(lib, fn)(DEV, ctypes.c_int64(n), ctypes.c_int64(n), DEV, None) == apsp.APSP_OK
    assert word(lib, "launches").value > 0 and word(lib, "programmatic").value == 0
