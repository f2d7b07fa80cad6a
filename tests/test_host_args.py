"""Host arguments of the calls as the C boundary gets them: poses and vectors of any layout and type as
row-major float64 bytes, too short ones refused, and a given stream by its handle."""
import numpy as np
import pytest

from paper_2309_16818_gb300 import mem as M


def _as_f64(b):
    return np.frombuffer(b, np.float64)


def test_poses_of_any_layout():
    T = np.arange(16.0).reshape(4, 4) + 0.25
    wide = np.zeros((4, 8))
    wide[:, ::2] = T
    for a in (T, T.astype(np.float32), np.asfortranarray(T), wide[:, ::2], T.tolist(), T.reshape(16)):
        assert np.array_equal(_as_f64(M._pose(a)), T.reshape(16))
    assert np.array_equal(_as_f64(M._pose(T.T)), T.T.reshape(16))
    B = np.stack([T, T + 1, T + 2])
    assert np.array_equal(_as_f64(M._pose(B[::-1], 3)), B[::-1].reshape(48))


@pytest.mark.parametrize("bad", [np.eye(3), np.zeros((3, 4)), np.zeros((2, 4, 4))])
def test_poses_of_another_size_are_refused(bad):
    with pytest.raises(ValueError):
        M._pose(bad)


def test_vectors():
    assert np.array_equal(_as_f64(M._f64((1, 2.5), 2)), [1.0, 2.5])
    assert np.array_equal(_as_f64(M._f64(np.arange(6.0)[::2], 2))[:2], [0.0, 2.0])
    assert np.array_equal(_as_f64(M._f64(np.float32([420, 421, 3, 4]), 4)), [420, 421, 3, 4])
    with pytest.raises(ValueError):
        M._f64((1.0,), 2)


def test_a_given_stream_is_passed_by_its_handle():
    class S:
        cuda_stream = 0x7F00_1234_5678
    assert M._stream(S()) == S.cuda_stream  # 64 bits: the calls declare pointer arguments
    for name in ("mem_fuse_pointcloud", "mem_fuse_image", "mem_get_layer", "mem_move_map", "mem_unet_forward"):
        assert getattr(M.lib(), name).argtypes[-1] is M.C.c_void_p, name
