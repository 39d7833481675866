"""The autotuners' cache file outlives a build: choices that another revision of the passes wrote
are timed again."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = ("from paper_1306_1821_gb300 import bps\n"
        "s = bps.Sampler(16, 100.0, 1, 2)\n"
        "print(bps.bps_x_pass_variant(s.ctx), bps.bps_z_line_pairs(s.ctx))\n"
        "s.close()\n")


def choices(path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", CODE], cwd=root, env=dict(os.environ, BPS_TUNE_CACHE=str(path)),
                         capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    return tuple(int(x) for x in out.stdout.split()[-2:]), json.loads(path.read_text())


def test_choices_of_another_revision_are_not_taken(tmp_path):
    import torch
    name = torch.cuda.get_device_name()
    path = tmp_path / "tune.json"
    old = {f"{p} N=16 chains=1 {what}": v for p in (name, name + " passes=0")
           for what, v in (("xleap", 6), ("zpairs", 16))}
    path.write_text(json.dumps(old))
    picked, cache = choices(path)
    new = {k: v for k, v in cache.items() if k not in old}
    assert sorted(k.rsplit(" ", 1)[1] for k in new) == ["xleap", "zpairs"]
    assert (next(v for k, v in new.items() if k.endswith("xleap")),
            next(v for k, v in new.items() if k.endswith("zpairs"))) == picked
    # this revision's own entries are taken as they stand
    path.write_text(json.dumps({k: {"xleap": 0, "zpairs": 16}[k.rsplit(" ", 1)[1]] for k in new}))
    assert choices(path)[0] == (0, 16)
