"""When the native marshaller counts as built (runs without a GPU)."""
import os

import torch

from paper_2606_12370_b200 import build as B


def test_the_marshaller_is_built_again_for_another_torch_or_python(monkeypatch):
    B.build_host()
    assert B._host_fresh()
    with monkeypatch.context() as m:
        m.setattr(torch, "__version__", torch.__version__ + ".other")
        assert not B._host_fresh()
    with monkeypatch.context() as m:
        m.setattr(B.sysconfig, "get_config_var", lambda name: "cpython-399-other")
        assert not B._host_fresh()
    with monkeypatch.context() as m:
        m.setattr(B, "HOST_FOR", os.path.join(B.HERE, "no such file"))
        assert not B._host_fresh()
    assert B._host_fresh()
