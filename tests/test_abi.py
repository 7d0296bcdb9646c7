"""CPU-side checks of the C ABI: the library builds, loads and exports every
function include/hgrms.h declares; argument errors are reported without any
device work; the binding fails loudly when the library is absent."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "include", "hgrms.h")


@pytest.fixture(scope="module")
def lib():
    from paper_1306_5390_gb300 import build, hgrms
    build.build()
    return hgrms.load_library()


def declared_functions():
    text = open(HEADER).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(hgrms_[a-z_]+)\s*\(", text)))


def test_header_declares_the_boundary():
    names = declared_functions()
    for must in ("hgrms_create", "hgrms_denoise", "hgrms_denoise_batch", "hgrms_destroy"):
        assert must in names


def test_every_declared_symbol_is_exported(lib):
    from paper_1306_5390_gb300 import hgrms
    out = subprocess.run(["nm", "-D", "--defined-only", hgrms.LIB_PATH], capture_output=True,
                         text=True, check=True).stdout
    exported = set(re.findall(r"\bT (hgrms_\w+)", out))
    for name in declared_functions():
        assert name in exported, name
        assert hasattr(lib, name)
    assert set(hgrms.EXPORTED) == set(declared_functions())
    # Nothing but the ABI leaks out of the library.
    assert not [s for s in re.findall(r"\bT (\w+)", out) if s.startswith("_ZN2hg")]


def test_strerror(lib):
    from paper_1306_5390_gb300 import hgrms
    assert hgrms.strerror(0) == "success"
    for code in (-1, -2, -3, -4, -5, -6, -7, -8):
        assert hgrms.strerror(code) not in ("success", "unknown error")
    assert hgrms.strerror(-99) == "unknown error"


def test_null_handle_errors_without_device_work(lib):
    from paper_1306_5390_gb300 import hgrms
    buf = (ctypes.c_uint8 * 16)()
    assert lib.hgrms_denoise(None, ctypes.addressof(buf), 4, 4, 10, 1, 5) == hgrms.HGRMS_EINVAL
    assert lib.hgrms_converged(None) == hgrms.HGRMS_EINVAL
    assert lib.hgrms_set_option(None, 1, 0) == hgrms.HGRMS_EINVAL
    assert lib.hgrms_last_cuda_error(None) == hgrms.HGRMS_EINVAL
    st = hgrms.hgrms_stats_t()
    assert lib.hgrms_stats(None, ctypes.byref(st)) == hgrms.HGRMS_EINVAL
    assert lib.hgrms_create(None, 0, None) == hgrms.HGRMS_EINVAL
    lib.hgrms_destroy(None)  # accepted
    ks = [0]
    assert hgrms.hgrms_denoise_batch(None, [ctypes.addressof(buf)], [4], [4], 10, 1, 5, ks) == hgrms.HGRMS_EINVAL
    assert lib.hgrms_denoise_async(None, ctypes.addressof(buf), 4, 4, 10, 1, 5) == hgrms.HGRMS_EINVAL
    assert lib.hgrms_wait(None) == hgrms.HGRMS_EINVAL


def test_kernel_table(lib):
    from paper_1306_5390_gb300 import hgrms
    for beta in range(1, 8):
        t = hgrms.hgrms_default_passes(beta)
        assert t >= 1 and hgrms.hgrms_has_kernel(beta, t) == 1
        assert hgrms.hgrms_has_kernel(beta, 1) == 1
    assert hgrms.hgrms_default_passes(0) == hgrms.HGRMS_EINVAL
    assert hgrms.hgrms_default_passes(8) == hgrms.HGRMS_EINVAL
    assert hgrms.hgrms_has_kernel(8, 1) == 0
    assert hgrms.hgrms_has_kernel(3, 4) == 0  # halo T*beta = 12 exceeds the tile margin


def test_no_gpu_is_reported_not_hidden(lib):
    import torch
    if torch.cuda.is_available():
        pytest.skip("a GPU is present")
    from paper_1306_5390_gb300 import hgrms
    h = ctypes.c_void_p()
    assert lib.hgrms_create(ctypes.byref(h), 0, None) == hgrms.HGRMS_ENODEV
    assert h.value is None
    with pytest.raises(hgrms.HgrmsError):
        hgrms.Denoiser(0)


def test_missing_library_fails_loudly(tmp_path, monkeypatch):
    from paper_1306_5390_gb300 import hgrms
    monkeypatch.setattr(hgrms, "_lib", None)
    with pytest.raises(RuntimeError, match="not built"):
        hgrms.load_library(str(tmp_path / "nope.so"))


def test_server_without_device(lib):
    """Creating a server needs a CUDA device (ENODEV here); bad arguments
    are rejected first."""
    import ctypes
    from paper_1306_5390_gb300 import hgrms
    h = ctypes.c_void_p()
    assert lib.hgrms_server_create(None, 0, 1 << 30, 2) == hgrms.HGRMS_EINVAL
    assert lib.hgrms_server_create(ctypes.byref(h), 0, 1 << 30, 0) == hgrms.HGRMS_EINVAL
    rc = lib.hgrms_server_create(ctypes.byref(h), 0, 1 << 30, 2)
    try:
        import torch
        has_gpu = torch.cuda.is_available()
    except ImportError:
        has_gpu = False
    if not has_gpu:
        assert rc == hgrms.HGRMS_ENODEV and not h.value
    else:
        assert rc == hgrms.HGRMS_OK
        lib.hgrms_server_destroy(h)
    lib.hgrms_server_destroy(None)  # accepted
    assert lib.hgrms_server_wait(None, 1, 0.0, None) == hgrms.HGRMS_EINVAL
    assert lib.hgrms_server_fail_allocations(None, 1) == hgrms.HGRMS_EINVAL


def test_header_constants_match_the_binding():
    """Every #define HGRMS_* integer constant of the header has the same value
    in the Python binding."""
    from paper_1306_5390_gb300 import hgrms
    text = open(HEADER).read()
    found = 0
    for name, val in re.findall(r"#define\s+(HGRMS_[A-Z0-9_]+)\s+\(?(-?\d+)\)?\s", text):
        assert getattr(hgrms, name) == int(val), name
        found += 1
    m = re.search(r"#define\s+HGRMS_NOALLOC_SCRATCH_BYTES\s+\((\d+)u << (\d+)\)", text)
    assert m and hgrms.HGRMS_NOALLOC_SCRATCH_BYTES == int(m.group(1)) << int(m.group(2))
    assert found >= 20


def test_batch_marshalling_matches_the_single_image_checks():
    """The batch loop gives the pointers and sizes of _ptr_shape and refuses
    what it refuses, for numpy arrays and tensors in any order; a null pointer
    stays one."""
    torch = pytest.importorskip("torch")
    from paper_1306_5390_gb300 import hgrms
    one = hgrms.Denoiser._ptr_shape
    a, t = np.zeros((3, 5), np.uint8), torch.zeros((4, 6), dtype=torch.uint8)
    imgs = [a, t, t[1:], np.zeros((0, 4), np.uint8), t.view(2, 12)]
    ptrs, rows, cols = hgrms.Denoiser._ptrs_shapes(imgs)
    assert list(zip(ptrs, rows, cols)) == [one(i) for i in imgs]
    P, R, C = hgrms._image_arrays(ptrs[:2] + [None], rows[:3], cols[:3])
    assert list(P) == [a.ctypes.data, t.data_ptr(), None] and list(R) == [3, 4, 3] and list(C) == [5, 6, 6]
    for bad in (t.t(), t.float(), torch.zeros(3, dtype=torch.uint8), np.zeros((2, 2)), a.T, torch.zeros((2, 2, 2), dtype=torch.uint8)):
        with pytest.raises(ValueError):
            one(bad)
        with pytest.raises(ValueError):
            hgrms.Denoiser._ptrs_shapes([t, bad])


class FakeLibrary:
    """Records the images of a batch call."""

    def hgrms_denoise_batch(self, h, P, R, C, n, alpha, beta, max_k, K):
        self.images = list(P), list(R), list(C), n
        return 0


def test_raw_batch_call_converts_as_ctypes_does(monkeypatch):
    """The raw call takes and refuses what ctypes arrays of the images' pointers
    and sizes take and refuse."""
    from paper_1306_5390_gb300 import hgrms
    lib = FakeLibrary()
    monkeypatch.setattr(hgrms, "load_library", lambda: lib)

    def call(ptrs, rows, cols):
        return hgrms.hgrms_denoise_batch(None, ptrs, rows, cols, 10, 1, 5, [0] * len(ptrs))
    assert call([ctypes.c_void_p(64), None, 80], (r for r in (1, ctypes.c_int(2), 3)), (4, True, 6)) == 0
    assert lib.images == ([64, None, 80], [1, 2, 3], [4, 1, 6], 3)
    call([64, -1], [1], [2 ** 32 + 5, 7])  # missing sizes are 0, which the library refuses
    assert lib.images == ([64, ctypes.c_void_p(-1).value], [1, 0], [5, 7], 2)
    call([], [], [])
    assert lib.images == ([None], [0], [0], 0)
    for ptrs, rows, cols in (([64], [1, 2], [3]), ([64], [1], [3, 4])):
        with pytest.raises(IndexError):
            call(ptrs, rows, cols)
    for ptrs, rows, cols in ((["64"], [1], [3]), ([64], [1.0], [3])):
        with pytest.raises(TypeError):
            call(ptrs, rows, cols)


def test_batch_sizes_past_32_bits_reach_the_library_as_a_single_images_do():
    from paper_1306_5390_gb300 import hgrms
    P, R, C = hgrms._image_arrays([64, 80], [1, 2], [2 ** 32 + 5, 2 ** 31])
    assert (list(P), list(R), list(C)) == ([64, 80], [1, 2], [5, -2 ** 31])
