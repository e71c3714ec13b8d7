"""Every FP32 triplet energy is added with compensation: no kernel of the force path adds
them to a plain float.  (The sources are read: the sums' errors are below those of the
terms, so no result shows the difference.)"""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2510_21230_gb300", "csrc")


def test_triplet_energies_go_to_compensated_sums():
    with open(os.path.join(CSRC, "atm_fwd.cuh")) as f:
        fwd = f.read()
    assert re.search(r"Sum<float> es;", fwd) and re.search(r"es\.add\(q3 \*", fwd)
    assert not re.search(r"float es\b", fwd)
    for name in ("atm_prod.cuh", "atm_owner.cuh"):
        with open(os.path.join(CSRC, name)) as f:
            src = f.read()
        assert re.search(r"Sum<R> esum", src) and "esum.add(uu)" in src, name
