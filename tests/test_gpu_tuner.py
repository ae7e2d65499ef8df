"""The slab-width tuner times plans: for a small problem a decode call would run
another kernel than the plan that the width is for."""
import json

import pytest

from synthetic import preset_graph

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def mld():
    import paper_1711_01783_gb300 as m
    return m


def test_widths_are_timed_in_plans(mld, tmp_path, monkeypatch):
    from paper_1711_01783_gb300.tune import WIDTHS, DecoderTuner, SlabWidthTuner
    g = mld.Graph.from_edges(preset_graph(0.1, 4096, 3))
    one_launch = []

    class Spy(mld.Decoder):
        def close(self):
            if getattr(self, "_h", None):
                one_launch.append(self.one_launch_decodes())
            super().close()

    monkeypatch.setattr(mld, "Decoder", Spy)
    path = tmp_path / "tune.json"
    # a choice made with decode calls, under the key it had then, is not taken over
    old = f"{g.signature}|9|f16|{torch.cuda.get_device_name()}"
    path.write_text(json.dumps({old: {"W": 64, "ms": {}}}))
    tuner = SlabWidthTuner(str(path))
    W = tuner.choose(g, 9, "f16")
    times = tuner.trials[tuner._key(g, 9, "f16")]
    assert set(times) == set(WIDTHS) and W == min(times, key=times.get)
    assert one_launch == [0] * len(WIDTHS)
    again = SlabWidthTuner(str(path))
    assert again.choose(g, 9, "f16") == W and not again.trials
    assert DecoderTuner()._key(g, 9, "f16") == "dec|" + old  # its own choices stay valid
