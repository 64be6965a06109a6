"""Rules that hold for the text of the CUDA sources (no GPU needed)."""
import pathlib
import re

import paper_1204_2280_gb300 as B

CSRC = pathlib.Path(B.__file__).parent / "csrc"


def _code(path):
    return re.sub(r"//[^\n]*", "", path.read_text())


def test_no_read_only_loads_in_overlapping_launches():
    """A kernel that is set up while its predecessor still runs may be
    resident while its inputs are written, so its file reads nothing through
    the read-only path: no restrict-qualified pointers, no __ldg or
    ld.global.nc, and nothing of the cache-hinted loads that a compiler may
    take for pure functions of their address."""
    found = []
    for path in sorted(CSRC.glob("*.cu")):
        code = _code(path)
        if "griddepcontrol" not in code and "ProgrammaticStreamSerialization" not in code:
            continue
        found.append(path.name)
        for word in ("__restrict__", "__ldg", "__ldcg", "__ldcs", "__ldca", "ld.global.nc"):
            assert word not in code, (path.name, word)
    assert found == ["k_msort.cu"]


def test_barrier_between_arrival_and_root():
    """A root's children are acquired by one lane and read by its whole warp:
    a warp barrier, which alone orders memory between lanes, stands between
    the arrival on the parent and the work on the roots."""
    code = _code(CSRC / "k_moments.cu")
    arrival = code.index("atom_add_acq_rel_gpu(&a.cell_done")
    between = code[arrival:code.index("root_cell<REFIT>(", arrival)]
    assert "__syncwarp();" in between
