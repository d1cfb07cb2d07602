"""bchar_destroy gives back everything that a handle holds, the buffers that only some
steps need included."""
import re
import os

import pytest

from paper_1908_05834_gb300 import inputs

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1908_05834_gb300", "csrc")


def _members(text, start):
    body = text[text.index(start):]
    body = body[:body.index("\n};")]
    return {n.split("[")[0].strip() for m in re.finditer(r"(?:bchar::)?Buf ([^;]+);", body) for n in m.group(1).split(",")}


def test_every_buffer_is_released():
    with open(os.path.join(CSRC, "internal.cuh")) as f:
        internal = re.sub(r"//.*", "", f.read())
    with open(os.path.join(CSRC, "capi.cu")) as f:
        capi = f.read()
    with open(os.path.join(CSRC, "amg.cu")) as f:
        amg = f.read()
    destroy = capi[capi.index("void bchar_destroy"):capi.index("bchar_status bchar_create_mesh")]
    handle = _members(internal, "struct bchar_mesh_s")
    assert len(handle) > 50
    assert {n for n in handle if not re.search(r"m->%s\b" % n, destroy)} == set()
    solver = _members(internal, "struct Amg")
    assert len(solver) > 20
    given = amg[amg.index("void amg_release"):]
    assert {n for n in solver if not re.search(r"A\.%s\b" % n, given)} == set()


@pytest.mark.gpu
def test_rows_wider_than_the_slab_are_given_back():
    import torch
    from paper_1908_05834_gb300 import build
    build.build()
    from paper_1908_05834_gb300 import bchar
    wl = inputs.workload("vortex2d_32", n=256)
    c = torch.tensor(wl.c0, dtype=torch.float64, device="cuda")
    out = torch.empty_like(c)
    free = []
    for _ in range(6):
        with bchar.Mesh(wl.coords, wl.phi, bchar.default_options(slab_width=1, qp_max_refine=0)) as mesh:
            mesh.set_velocity(wl.faces(0))
            info = mesh.step(0.01, c, out)
            assert info["spill_rows"] > 50000
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])
    # 2.5 MB and more of each handle's spill area stayed on the device
    assert free[1] - free[-1] < 4 << 20, free
