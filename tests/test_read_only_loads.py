"""The kernels of a step overlap (programmatic dependent launch): each is resident while its
predecessor still writes, so the read-only path (__ldg, ld.global.nc), defined for data that
nothing writes during a kernel's whole lifetime, may read weights and tables only.  Every
use of it in the sources is checked against the weights' names (no GPU needed)."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2609_29505_gb300" / "csrc"

# gains, shifts, embeddings, positions, projection weights; wp, w and W are pointers into w_stem,
# and into GemvParams::W / w_seg, where they are used
WEIGHTS = re.compile(r"^(?:reinterpret_cast<const uint[24]\*>\()?(?:p\.(?:g|b|embed|pos|W)\b|wp \+|w \+|W \+)")


def _arguments(text):
    for m in re.finditer(r"__ldg\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        yield text[m.end():i - 1]


def test_read_only_loads_read_weights_only():
    found = 0
    for path in sorted(list(CSRC.glob("*.cu")) + list(CSRC.glob("*.cuh")) + list(CSRC.glob("*.h"))):
        code = re.sub(r"//[^\n]*", "", path.read_text())
        assert "ld.global.nc" not in code and "__restrict__" not in code, path.name
        for arg in _arguments(code):
            found += 1
            assert WEIGHTS.match(arg), (path.name, arg)
    assert found >= 8
