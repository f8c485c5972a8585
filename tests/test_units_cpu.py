"""Where the special-function unit's approximate reciprocals may stand: in the
marker and spread kernels' closed form only.  The element forces and the whole
adjoint divide in IEEE arithmetic (their strains and second derivatives have no
approximate unit in front of them)."""
import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_1612_03399_gb300" / "csrc"


def code(name):
    return re.sub(r"//[^\n]*", "", (CSRC / name).read_text())


def test_forces_and_adjoint_divide_in_ieee():
    for name in ("force_elems.cuh", "k_force.cu", "k_adjoint.cu"):
        assert not re.search(r"__fdividef|rcp_fast|__frcp|rcp\.approx|div\.approx", code(name)), name
    # the adjoint's gradients ask for correctly rounded reciprocals
    assert not re.search(r"\bdir_grad\(", code("k_adjoint.cu"))
    hess = code("mls_closed_form.cuh").split("void dir_hess")[1].split("\n}\n")[0]
    assert "dir_grad<true>" in hess and "rcp_fast" not in hess
