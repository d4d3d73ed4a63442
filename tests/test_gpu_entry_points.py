"""smoke(), the entry point that shows a checkout to work on a GPU: it counts the launches of each block it runs."""
import pytest

pytestmark = pytest.mark.gpu


def test_smoke(capsys):
    import __graft_entry__
    __graft_entry__.smoke()
    assert "smoke ok" in capsys.readouterr().out
