"""A failing pbfb_charges_set never leaves a mesh that counts as having charges while their sums and positions are of two
sets or freed: refusals come before anything of the mesh is overwritten, and the mesh has no charges from the first
overwritten buffer on until all of them are there.  Checked on the source, on CPU (running out of device memory is
no test)."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_21713_gb300", "csrc",
                   "solver.cu")


def test_no_charges_while_they_change():
    body = re.search(r"^int charges_set\(.*?^}", open(SRC).read(), re.S | re.M).group(0)
    off, on = body.index("m->charges = false;"), body.rindex("m->charges = true;")
    refusals = [m.start() for m in re.finditer(r"PBFB_ERR_INVALID|charge_outside\(|point_load\(", body)]
    overwritten = [m.start() for m in re.finditer(r"m->(?:rho|qxyz|qz|coul)\b|m->nq = |launch_coulomb\(", body)]
    assert refusals and overwritten
    assert max(refusals) < off < min(overwritten) and max(overwritten) < on
    assert body.index("cudaStreamSynchronize") < on
