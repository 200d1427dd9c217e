"""The autotuner's choice for a recomputing backward (what captured graphs run) is
kept apart from the one for the options' default backward."""
import json

import numpy as np
import pytest

from paper_2205_14330_gb300 import scenes

pytestmark = pytest.mark.gpu


def test_a_choice_per_backward(tmp_path):
    import __graft_entry__ as g
    g.build()
    from paper_2205_14330_gb300 import pbr
    rng = np.random.default_rng(2)
    n = 2000
    sc = pbr.Scene(rng.uniform(-0.5, 0.5, (n, 3)).astype(np.float32),
                   scenes.sh_coeffs(rng, n, 1, std=0.2), np.full(n, 0.5, np.float32),
                   np.full(n, 0.03, np.float32), 1)
    cams = [scenes.camera((0.0, 0.3, 2.5), 64, 48)]
    R = pbr.Renderer(0)
    pbr.autotune(R, sc, cams, reps=1)
    R.save_tuning(tmp_path / "a.json")
    data = json.loads((tmp_path / "a.json").read_text())
    assert [c["mode"] for c in data["classes"]] == [1]
    data["classes"][0].update(tile_w=8, tile_h=8, batch_depth=512, persistent=0)
    (tmp_path / "b.json").write_text(json.dumps(data))
    assert R.load_tuning(tmp_path / "b.json") == 1

    def choice(R, bwd_mode):
        info = {}
        o, _ = pbr.autotune(R, sc, cams, pbr.default_opts(bwd_mode=bwd_mode), reps=1,
                            report=False, info=info)
        return (o.tile_w, o.tile_h, o.batch_depth, o.persistent), info["n_timed"]

    assert choice(R, 0) == ((8, 8, 512, 0), 0)  # the file's
    picked, timed = choice(R, 1)
    assert timed == pbr.N_TUNE_CANDIDATES
    assert choice(R, 1) == (picked, 0) and choice(R, 0) == ((8, 8, 512, 0), 0)
    R.save_tuning(tmp_path / "c.json")
    R2 = pbr.Renderer(0)
    assert R2.load_tuning(tmp_path / "c.json") == 2
    assert choice(R2, 1) == (picked, 0) and choice(R2, 0) == ((8, 8, 512, 0), 0)
    R2.close()
    R.close()
