"""PDN_PDL=0 launches every kernel plainly: one helper sets the attribute of
programmatic dependent launch, and runs with and without it are equal bit for
bit, the learned law's kernel and its training included."""
import os
import re
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2301_05552_gb300", "csrc")


def test_one_helper_sets_the_attribute():
    naming = {n for n in os.listdir(CSRC) if "ProgrammaticStreamSerialization" in open(os.path.join(CSRC, n)).read()}
    assert naming == {"pdn_launch.h"}
    helper = open(os.path.join(CSRC, "pdn_launch.h")).read()
    assert re.search(r'getenv\("PDN_PDL"\)', helper) and re.search(r"numAttrs = pdl_on\(\) \? 1 : 0", helper)


CHILD = r"""
import sys
import numpy as np
import paper_2301_05552_gb300 as pkg
import pdn_inputs as pi
w = pi.damage_fp32_plate(nx=33, ny=27, plies=6, Lx=16.5, Ly=13.5, H=1.65)
st = pi.seeded_state(w.plate, 7, amp=0.02, vamp=300.0, dimple=(8.25, 6.75, 0.12, 3.0))
law = pkg.pdn_sur_create(w.material, 0.41, seed=0)
pkg.pdn_sur_generate(law, 4000, 8, 0.01, 0.4, 0.9, seed=1)
loss = pkg.pdn_sur_train(law, 200, 1024, 2e-3, seed=2)
params, scaling = pkg.pdn_sur_get_params(law)
out = dict(loss=loss, params=params, scaling=scaling)
for name in ("exact", "learned"):
    s = pkg.Solver(w)
    if name == "learned":
        pkg.pdn_set_surrogate(s.ctx, law, 0.9)
    pkg.pdn_set_state(s.ctx, *st)
    s.step(100)
    out[name + "_d"], out[name + "_v"], _ = s.state()
    out[name + "_h"], out[name + "_r"] = pkg.pdn_get_history(s.ctx)
    s.close()
np.savez(sys.argv[1], **out)
"""


@pytest.mark.gpu
def test_plain_launches_give_the_same_bits(tmp_path):
    import numpy as np
    res = []
    for pdl in ("1", "0"):
        f = str(tmp_path / f"pdl{pdl}.npz")
        env = dict(os.environ, PDN_PDL=pdl, PDN_HEX_VARIANT="0", PYTHONPATH=ROOT)
        subprocess.run([sys.executable, "-c", CHILD, f], env=env, cwd=ROOT, check=True, timeout=300)
        res.append(np.load(f))
    assert set(res[0].files) == set(res[1].files) and np.abs(res[0]["learned_d"]).max() > 0.0
    for k in res[0].files:
        assert np.array_equal(res[0][k], res[1][k]), k
