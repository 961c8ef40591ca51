"""The autotuner on a runner whose knobs size nothing: its defaults, timed
once per phase, whatever noise the other choices or an older cache show."""
import json

from paper_2510_10256_gb300.tune import Autotuner


class InertRunner:
    tuning_inert = True

    def __init__(self):
        self.knobs = {0: (2.0, 64), 1: (2.0, 64)}
        self.passes = 0

    def set_timing(self, on=True):
        pass

    def set_tuning(self, ph, f, b):
        self.knobs[ph] = (f, b)

    def stage_ms(self):  # noise that falls from pass to pass
        return [1.0 / self.passes, 0.0, 0.0, 2.0 / self.passes, 0.0]

    def run(self):
        self.passes += 1


def test_keeps_the_defaults(tmp_path):
    path = tmp_path / "tune.json"
    old = {"k": {str(ph): {"cell_factor": 4.0, "pair_block": 128, "stage_ms": 1.3, "default_ms": 1.4, "tried": 14}
                 for ph in (0, 1)}}
    path.write_text(json.dumps(old))
    r = InertRunner()
    c = Autotuner(str(path)).tune(r, "k", r.run)
    assert r.knobs == {0: (1.0, 256), 1: (1.0, 256)} and not c["cached"]
    for ph in "01":
        assert (c[ph]["cell_factor"], c[ph]["pair_block"], c[ph]["tried"]) == (1.0, 256, 1)
        assert c[ph]["stage_ms"] == c[ph]["default_ms"] > 0.0
    assert r.passes == 2 * 3
    assert json.loads(path.read_text()) == old


def test_the_librarys_scenes_say_so():
    from paper_2510_10256_gb300.contact import ContactBatch, ContactScene
    assert ContactScene.tuning_inert and ContactBatch.tuning_inert
