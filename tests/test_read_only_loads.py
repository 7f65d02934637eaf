"""Loads of the read-only path in the kernels' sources.  The kernels of a call start before the previous
one is complete and wait for it; a load that is promised not to change while its kernel runs may be moved
above that wait, so only the rig's constant tables are read that way: never the results of earlier launches
(collapsed levels, level-0 samples) and never frames, whose producer may be such a kernel too."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1810_03988_gb300", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))

# tables that are written when the rig (or batch) is created, by element type and name, and the shared-memory
# argument `a` of the EXPAND helpers
TABLES = {
    "float": {"d1w", "wcol"}, "float4": {"d1cols", "cols", "a"}, "int4": {"slots"},
    "int": {"camlist", "centers", "cam_slot_start", "need"},
}
TABLE_TYPES = {"CamDev", "CamRef", "D1Cams", "D1Rec", "D1Tile", "SoloTile", "Tile", "LevelTile", "UpTile", "BwTile",
               "BTask", "BatchRigDev", "R"}  # R: load_record's
LDG_OF = re.compile(r"(wp|wcol|m < D1_TY \? wp \+ D1_SX : wp|x\.wt)\b|reinterpret_cast<const uint4\*>\(p\)")


def _code(path):
    text = open(path).read()
    text = re.sub(r"/\*.*?\*/", " ", text, flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_only_constant_tables_take_the_read_only_path(path):
    code = _code(path)
    for typ, name in re.findall(r"const\s+(\w+)\s*\*\s*__restrict__\s+(\w+)", code):
        assert typ in TABLE_TYPES or name in TABLES.get(typ, ()), f"const {typ}* __restrict__ {name}"
    for m in re.finditer(r"__ldg\(", code):
        arg = code[m.end():m.end() + 80]
        assert LDG_OF.match(arg), f"__ldg({arg.splitlines()[0]}"
