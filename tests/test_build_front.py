"""When _front.so is built again."""
import torch

from paper_2511_09323_b200 import build as moc_build


def test_a_module_of_another_torch_is_not_current(monkeypatch):
    moc_build.build()
    assert moc_build._front_is_current()
    with monkeypatch.context() as m:
        m.setattr(torch, "__version__", "0.0.1")
        assert not moc_build._front_is_current()
    assert moc_build._front_is_current()
