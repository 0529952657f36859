"""Entries of the schedule cache file whose CTA shape does not admit the table's M are
not used: the call runs the default schedule, as without a file."""
import json
import os
import subprocess
import sys

import pytest
import torch

import paper_2511_14923_gb300 as gbs

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = "import sys, json; sys.path.insert(0, {root!r}); import paper_2511_14923_gb300 as gbs; " \
        "print(json.dumps(gbs.schedule({M}, 4, {prec!r})))"


def schedule_with(env_file, M, prec):
    env = {k: v for k, v in os.environ.items() if k != "GBS_AUTOTUNE_CACHE"}
    if env_file:
        env["GBS_AUTOTUNE_CACHE"] = str(env_file)
    out = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, M=M, prec=prec)], env=env, capture_output=True,
                         text=True)
    assert out.returncode == 0, out.stderr
    return json.loads(out.stdout)


@pytest.mark.parametrize("M,prec,variant,used", [(305, "fp32r", 2, True), (306, "fp32r", 2, False),
                                                 (673, "fp64", 4, True), (674, "fp64", 4, False),
                                                 (162, "fp32r", 9, False), (400, "fp64", 6, False)])
def test_shape_that_does_not_admit_m(tmp_path, M, prec, variant, used):
    gbs.build()
    maj, mnr = torch.cuda.get_device_capability(0)
    entry = {"cc": 10 * maj + mnr, "sms": torch.cuda.get_device_properties(0).multi_processor_count, "M": M, "kmax": 4,
             "precision": gbs.PRECISIONS[prec], "grain": 1, "ccap": 16, "variant": variant}
    f = tmp_path / "tune.json"
    f.write_text(json.dumps([entry]))
    got = schedule_with(f, M, prec)
    assert got == ({"variant": variant, "grain": 1, "ccap": 16} if used else schedule_with(None, M, prec))
