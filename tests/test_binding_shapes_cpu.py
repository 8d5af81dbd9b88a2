"""The binding takes a level's node counts from the library at every call: the check of a displacement's
size is the only one between a tensor and the kernels that read it."""
import ctypes

import numpy as np
import pytest

pytest.importorskip("torch")
reg = pytest.importorskip("paper_1812_06765_gb300")
from paper_1812_06765_gb300 import _lib  # noqa: E402


class _FakeLibrary:
    """reg_level_info of a handle whose images change: nodes[level], an error without a handle."""
    nodes = {0: (5, 6, 7), 1: (3, 4, 5)}

    def reg_level_info(self, h, level, m, n, sp, H):
        if h is None or level not in self.nodes:
            return -1
        n[0], n[1], n[2] = self.nodes[level]
        return 0

    def reg_last_error(self, h):
        return b"refused"

    def reg_destroy(self, h):
        return 0


def test_node_shape_follows_the_handle(monkeypatch):
    fake = _FakeLibrary()
    monkeypatch.setattr(_lib, "lib", lambda: fake)
    monkeypatch.setattr(reg, "_require_cuda", lambda: None)
    monkeypatch.setattr(_lib, "reg_create", lambda cfg, stream=None: ctypes.c_void_p(1234))
    r = reg.Registration(_lib.RegConfig(), stream=type("S", (), dict(cuda_stream=0)))
    assert r.node_shape(0) == (3, 7, 6, 5)
    assert r.node_shape(np.array(1)) == (3, 5, 4, 3)     # whatever int() takes is a level
    fake.nodes = {0: (9, 8, 7)}                          # other images, set through the C entry
    assert r.node_shape(0) == (3, 7, 8, 9)
    with pytest.raises(_lib.RegError):
        r.node_shape(1)
    r.close()
    with pytest.raises(_lib.RegError):                   # a closed handle is refused
        r.node_shape(0)
