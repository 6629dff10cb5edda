"""grid_specialize with every CUDA call failing in turn, on a CUDA runtime
without a GPU: the call reports the error and leaves no device memory behind,
whichever call fails."""
import pytest

from paper_2607_11951_gb300 import grid as G
from tests import fakes
from workloads import grammar_text


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fakes.link(tmp_path_factory.mktemp("fake"))


@pytest.mark.parametrize("ones", [0, 1])  # tables without walked or verdict-class spellings, and with
def test_every_failing_call_frees_everything(fake, ones):
    with fakes.use(fake) as rt:
        g = G.Grammar(grammar_text("sql"), [], {"TABLE_NAME": ["t1"], "COLUMN_NAME": ["c1", "c2"]})
        toks = [bytes([b]) for b in range(256)] + [b"<eos>"]
        v = G.Vocab(toks, 256, [])
        rt.reset(ones=ones)
        s = G.Spec(g, v)
        calls, kept = rt.get("calls"), rt.get("live")
        del s
        assert rt.get("live") == 0 and kept > 0 and calls > 40
        for k in range(1, calls + 1):
            rt.reset(fail_at=k, ones=ones)
            with pytest.raises(G.GridError) as e:
                G.Spec(g, v)
            assert e.value.code == -7
            del e
            assert rt.get("live") == 0, (k, rt.get("live"))
        rt.reset(ones=ones)
        s = G.Spec(g, v)
        assert rt.get("live") == kept
        del s, g, v
