"""The smoke hook runs to its end on a GPU: launches counted, result within the FP64-grade bound of the oracle's."""
import pytest

pytestmark = pytest.mark.gpu


def test_smoke_hook(capsys):
    import __graft_entry__
    __graft_entry__.smoke()
    assert "bit-identical = True" in capsys.readouterr().out
