"""What a GPU run cannot show, read from the CUDA sources: memory that one lane of a warp writes and
another reads has a barrier between the two (shuffles order no memory)."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1106_0322_gb300", "csrc")


def _code(name):
    src = open(os.path.join(CSRC, name)).read()
    src = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
    return re.sub(r"//[^\n]*", "", src)


def _body(src, head):
    """The text of the function whose declaration starts with `head`, braces included."""
    at = src.index("{", src.index(head))
    depth = 0
    for k in range(at, len(src)):
        depth += {"{": 1, "}": -1}.get(src[k], 0)
        if depth == 0:
            return src[at : k + 1]
    raise AssertionError(head)


def test_mala_gradient_row_is_ordered_between_the_lanes_that_write_and_read_it():
    """mala_reverse stores coordinate j of a proposal's gradient from lane j % 32 when p % 4 != 0; the
    move kernel then reads an accepted row from lane (j / 4) % 32 of the same warp."""
    assert any(j % 32 != (j // 4) % 32 for j in range(5))
    src = _code("k_smc.cu")
    rev, move = _body(src, "__device__ __forceinline__ FSum mala_reverse"), _body(src, "k_move_mala(MoveArgs a")
    store = rev.index("g1[j] = ")
    after_store = rev[store:]
    between = move[move.index("mala_reverse<") : move.index("gsrc[j]")]
    assert re.search(r"__syncwarp\(\)|__syncthreads\(\)", after_store + between)


def test_mala_drift_is_rounded_as_written_in_both_densities():
    """The slope in MALA's drift comes from functions whose every operation names its rounding, in the
    reverse density and in the forward one, instead of from a sum that the compiler may contract."""
    src = _code("k_smc.cu")
    drifts = re.findall(r"const float drift = [^;]*;", src)
    assert len(drifts) == 5
    assert [bool(re.search(r"\* slope_reverse\([^;]*\);$", d)) for d in drifts] == [True] * 3 + [False] * 2
    assert [bool(re.search(r"\* slope_forward\([^;]*\);$", d)) for d in drifts] == [False] * 3 + [True] * 2
    for name in ("slope_forward(", "slope_reverse("):
        body = _body(src, "__device__ __forceinline__ float " + name)
        assert re.search(r"__f(maf|add)_rn\(", body)
        assert not re.search(r"[^_a-z] [+*/-] |__fdividef", body)
