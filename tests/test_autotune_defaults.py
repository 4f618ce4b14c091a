"""The tuner's grid holds the library's defaults: a call that sets no knob may take the small-graph kernels,
which a tuned option must not cost it."""
import json

import graphgen as gg
from paper_1509_08267_gb300 import Options, autotune


def _default(cfg):
    return autotune._options(cfg, timing=False) == Options()


def test_the_grid_holds_the_defaults():
    seen = []

    def timer(cfg):
        seen.append(cfg)
        return 0.1 if _default(cfg) else 1.0

    best = autotune.tune({"uniform-small": timer}, log=lambda *_: None)["uniform-small"]
    assert sum(map(_default, seen)) == 1
    assert _default(best)


def test_a_default_entry_gives_the_defaults(tmp_path):
    best = autotune.tune({"uniform-small": lambda cfg: 0.1 if _default(cfg) else 1.0}, log=lambda *_: None)
    path = tmp_path / "t.json"
    path.write_text(json.dumps(best))
    g = gg.er(3000, 12.0, 1)
    assert autotune.options_for(g.n, g.degrees(), str(path)) == Options()


def test_whole_calls_are_timed(monkeypatch):
    asked = []

    def color(rowptr, colidx, mode, seed, options):
        asked.append(options)

    monkeypatch.setattr(autotune, "color", color)
    cfg = {"small_max_degree": 0, "chunk": 0, "blocks_per_sm": 0, "compact": True, "core_vertices": 0}
    assert autotune.time_config(None, None, cfg, repeats=3) >= 0.0
    assert len(asked) == 4 and all(o == Options() for o in asked)  # (no flag that keeps a call off a path)
