"""Workspace sizes of few-channel layers whose stride is beyond what the tensor-core engine's operand copies reach: the
CUDA-core engine reads the caller's tensors, so the query has room for the header, the int32 sums and (update calls) the
scratch gradient, and nothing is widened or padded."""
import ctypes

import pytest

OP_CONV_FWD, OP_CONV_WGRAD, OP_CONV_WGRAD_UPDATE = 2, 4, 7
HEADER = 256 * 1024


def _up(v):
    return (v + 255) // 256 * 256


@pytest.fixture(scope="module")
def query():
    from paper_2009_13108_b200 import build
    lib = ctypes.CDLL(build.build())
    lib.niti_workspace_bytes.restype = ctypes.c_size_t

    def call(op, *dims):
        return lib.niti_workspace_bytes(op, (ctypes.c_int64 * len(dims))(*dims), len(dims))
    return call


@pytest.mark.parametrize("B,H,W,Ci,Co,R,pad,stride", [
    (64, 224, 224, 3, 768, 16, 0, 16), (64, 224, 224, 3, 768, 14, 0, 14), (8, 90, 70, 1, 24, 9, 2, 9),
    (2, 60, 60, 12, 33, 12, 3, 12)])
def test_nothing_is_copied_above_stride_8(query, B, H, W, Ci, Co, R, pad, stride):
    dims = (B, H, W, Ci, Co, R, R, pad, stride)
    Ho, Wo = (H + 2 * pad - R) // stride + 1, (W + 2 * pad - R) // stride + 1
    grad = Co * R * R * Ci
    assert query(OP_CONV_FWD, *dims) == HEADER + _up(4 * B * Ho * Wo * Co)
    assert query(OP_CONV_WGRAD, *dims) == HEADER + _up(4 * grad)
    assert query(OP_CONV_WGRAD_UPDATE, *dims) == HEADER + _up(4 * grad) + _up(grad)


def test_windows_have_room_for_the_widened_image(query):
    dims = (64, 224, 224, 3, 96, 11, 11, 2, 4)
    assert query(OP_CONV_WGRAD, *dims) >= HEADER + 4 * 96 * 11 * 11 * 3 + 64 * 224 * 224 * 4
