"""Register splits between warp roles, checked on the sources (no GPU).  The four warps of a warpgroup have to execute
the same setmaxnreg instruction.  A kernel whose roles end inside a warpgroup (11 gridding warps and the issuer of
the tensor-core form at N_p = 128) satisfies that with one instruction per register count, in a branch that whole
warpgroups take."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1510_08318_gb300", "csrc")


def test_one_instruction_per_register_count():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        with open(path) as f:
            found = re.findall(r'"setmaxnreg\.(?:inc|dec)[^;]*;"\s*::\s*"n"\((\w+)\)', f.read())
        assert len(found) == len(set(found)), (path, found)


def test_roles_of_the_tensor_core_form():
    """The instructions lie on a branch that parts the warps at a whole warpgroup, before the last group's roles part."""
    with open(os.path.join(CSRC, "moff_dftgemm.cu")) as f:
        src = f.read()
    const = {k: int(v) for k, v in re.findall(r"constexpr int (NXW|NGW) = (\d+);", src)}
    assert const["NXW"] % 4 == 0 and (const["NGW"] + 1) % 4 == 0
    lines = [s.strip() for s in src.split("\n")]
    lines = [s for s in lines if s and not s.startswith("//")]
    inc, = [i for i, s in enumerate(lines) if "setmaxnreg.inc" in s]
    dec, = [i for i, s in enumerate(lines) if "setmaxnreg.dec" in s]
    assert lines[inc - 1] == "if (warp < NXW) {"
    assert lines[dec - 1] == "} else {" and lines[dec + 1] == "if (warp < NXW + NGW) {"
