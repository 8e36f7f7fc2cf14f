"""Host side of the Python binding that needs no GPU."""
import ctypes
import types
import warnings

import numpy as np
import pytest

from paper_2503_08217_gb300 import binding


def _camera(w):
    cam = types.SimpleNamespace(width=16, height=8, fx=9.0, fy=9.0, cx=8.0, cy=4.0, near=0.2, world_to_cam=w)
    return np.array(binding.make_camera(cam).world_to_cam)


BASE = np.random.default_rng(1).standard_normal((3, 4))


@pytest.mark.parametrize("w", [
    BASE.astype(np.float32), BASE, BASE.astype(np.float16), BASE.astype(">f4"), BASE.tolist(),
    np.asfortranarray(BASE.astype(np.float32)), np.repeat(BASE.astype(np.float32).reshape(-1), 2)[::2],
    BASE.astype(np.float32).T.copy().T, (100 * BASE).astype(np.int64), BASE > 0, BASE.astype(object),
    np.full((3, 4), 1e300), np.full((3, 4), (1 << 54) + 3), np.full((3, 4), "1.5"),
    np.full((3, 4), np.longdouble(1) + np.longdouble(2) ** -24 + np.longdouble(2) ** -60)],
    ids=["f4", "f8", "f2", "swapped", "list", "fortran", "strided", "transposed", "int", "bool", "object",
         "overflow", "wide_int", "text", "longdouble"])
def test_camera_matrix_takes_what_float_takes(w):
    """Every entry is float(x) rounded to 32 bits, without a warning."""
    want = np.array((ctypes.c_float * 12)(*[float(x) for x in np.asarray(w).reshape(12)]))
    with warnings.catch_warnings():
        warnings.simplefilter("error")
        np.testing.assert_array_equal(_camera(w), want)


@pytest.mark.parametrize("w", [np.zeros((3, 4), "M8[s]"), np.zeros((4, 4)), [["a"] * 4] * 3, None])
def test_camera_matrix_refuses_the_rest(w):
    with pytest.raises((TypeError, ValueError)):
        _camera(w)


@pytest.mark.parametrize("raw", [True, False])
def test_current_stream_with_and_without_the_raw_handle(monkeypatch, raw):
    import torch
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=0x77))
    monkeypatch.setattr(binding, "_raw_stream", (lambda device: 0x70 + device) if raw else None)
    assert binding._stream() == (0x73 if raw else 0x77)
    assert binding._stream(types.SimpleNamespace(cuda_stream=5)) == 5
