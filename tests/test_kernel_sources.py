"""Rules of the kernel sources that no run can show: a warp-wide exchange that names
too few lanes is undefined, and may still give the right answer on one compiler."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2101_11552_gb300", "csrc")
FILES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))
# every warp exchange whose first argument is a lane mask
MASKED = r"__(?:shfl(?:_up|_down|_xor)?|ballot|any|all|match_any|match_all|reduce_\w+)_sync\s*\(\s*([^,]*),"


def code(path):
    text = re.sub(r"/\*.*?\*/", "", open(path).read(), flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def declared(statement):
    """Names that one constexpr declaration introduces (several after one type)."""
    return re.findall(r"\b(k[A-Z]\w*)\s*(?:=(?!=)|\{)", statement)


def test_every_warp_exchange_is_by_all_lanes():
    """One place names the mask, so that no name of a kernel's or a policy's own scope can
    stand in for it."""
    where = {os.path.basename(p): re.findall(MASKED, code(p)) for p in FILES}
    assert {name for name, masks in where.items() if masks} == {"common.cuh"}
    assert set(where["common.cuh"]) == {"kAllLanes"}
    assert re.search(r"constexpr unsigned kAllLanes = 0xffffffffu;", code(os.path.join(CSRC, "common.cuh")))


def test_no_class_constant_hides_a_namespace_constant():
    outer, inner = {}, {}
    for p in FILES:
        for line in code(p).split(";"):
            m = re.search(r"\n(\s*)(?:template\s*<[^<>]*>\s*)?(?:static\s+|inline\s+)?constexpr\b[^;]*$", line)
            if m:
                into = inner if m.group(1).strip("\n") else outer
                for name in declared(line[m.start():]):
                    into.setdefault(name, set()).add(os.path.basename(p))
    assert "kAllLanes" in outer and "kTile" in inner, "the scan finds the constants"
    hidden = {name: (sorted(outer[name]), sorted(inner[name])) for name in outer.keys() & inner.keys()}
    assert not hidden, hidden
