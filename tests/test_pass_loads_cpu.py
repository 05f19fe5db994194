"""Kernels launched programmatically dependent are resident while the grid before them writes, and a
non-coherent load (__ldg, or a const __restrict__ parameter) is defined only on memory that nothing
writes while its kernel runs. So such loads are left to tables that no pass writes; whatever the
passes hand on is read with plain loads, which also stay behind the wait."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_2606_01598_gb300" / "csrc"
FILES = sorted([*CSRC.glob("*.cu"), *CSRC.glob("*.cuh"), *CSRC.glob("*.h")])

# what __ldg may read: transforms' twiddles, the influence table, the network's radial weights
LDG = ("tw + ", "a.gtab + ", "row + ")
# const __restrict__ parameters of tables: twiddles, frame descriptors, species, offsets, parameters
TABLES = {"tw", "tz", "ty", "frames", "species", "offs", "WR", "P"}
# functions whose other const __restrict__ parameters are no pass data: shared memory; an ordinary launch
OTHER = {"fft_stage", "k_scale_signed"}
# kernels that follow the one that writes the parameters
AFTER_PARAMETERS = {"k_cast_weights", "k_adam"}


def _code(path):
    return re.sub(r"//[^\n]*", "", path.read_text())


def test_ldg_reads_tables_only():
    found = 0
    for path in FILES:
        for m in re.finditer(r"__ldg\(", _code(path)):
            arg = _code(path)[m.end():m.end() + 60]
            assert arg.startswith(LDG), (path.name, arg)
            found += 1
    assert found


def test_const_restrict_parameters_are_tables():
    found = 0
    for path in FILES:
        for m in re.finditer(r"(\w+)\(([^()]*__restrict__[^()]*)\)\s*\{", _code(path)):
            name, params = m.groups()
            for q in params.split(","):
                r = re.search(r"__restrict__\s+(\w+)", q)
                if not r or name in OTHER:
                    continue
                assert "const" in q and r.group(1) in TABLES, (path.name, name, q.strip())
                assert not (name in AFTER_PARAMETERS and r.group(1) == "P"), (path.name, name)
                found += 1
    assert found > 5


def test_no_restrict_locals():
    for path in FILES:
        for line in _code(path).splitlines():
            assert not re.search(r"__restrict__\s+\w+\s*=", line), (path.name, line.strip())
