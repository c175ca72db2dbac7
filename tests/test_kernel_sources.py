"""Rules of the kernels that a run need not show to be broken, checked in the sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_02947_b200", "csrc")


def _code():
    text = "".join(open(os.path.join(CSRC, f)).read() for f in sorted(os.listdir(CSRC)))
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def _closed(text, i, pair):
    """End of the bracket that opens at text[i]."""
    depth = 0
    while True:
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        i += 1
        if depth == 0:
            return i


def _function(code, name):
    """Parameters and body of the function of this name."""
    for m in re.finditer(r"\b" + name + r"\s*\(", code):
        end = _closed(code, m.end() - 1, "()")
        if code[end:].lstrip().startswith("{"):
            body = code.index("{", end)
            return code[m.end():end - 1], code[body:_closed(code, body, "{}")]
    raise AssertionError(f"{name} has no definition")


# A kernel that starts while its predecessor still writes waits before it reads.  That order holds for ordinary loads only: __ldg,
# and a load through a __restrict__ parameter, which the compiler may take for the read-only path, are for memory that nothing
# writes while the kernel is resident, and may be moved over the wait.
OVERLAPPED = ["atf_prefill_prep_kernel", "atf_split_prep_kernel", "atf_decode_kernel", "atf_decode_tiles_kernel", "atf_prefill_pipe_kernel",
              "atf_rope_kernel"]


@pytest.mark.parametrize("kernel", OVERLAPPED)
def test_reads_behind_the_wait_stay_there(kernel):
    code = _code()
    parameters, body = _function(code, kernel)
    assert "grid_dependency_wait()" in body
    for helper in ("atf_write_schedule", "merge_splits"):
        if helper in body:
            p, b = _function(code, helper)
            parameters, body = parameters + p, body + b
    assert "__restrict__" not in parameters
    assert "__ldg" not in body and "ld.global.nc" not in body


def test_every_overlapped_kernel_is_looked_at():
    """A kernel is launched either in the ordinary way or by one of the two calls that set the attribute."""
    code = _code()
    kernels = set(re.findall(r"\b(atf_\w+_kernel)\b", code))
    assert set(OVERLAPPED) == {k for k in kernels if not re.search(k + r"\s*<<<", code)}
    assert len(kernels) > len(OVERLAPPED) and len(re.findall(r"ProgrammaticStreamSerialization;", code)) == 2


def test_sums_are_read_behind_a_barrier_of_the_warp():
    """In turns one lane waits for a tile's sums and the whole warp reads them: a shuffle passes a value on, not the order of memory."""
    _, body = _function(_code(), "atf_prefill_pipe_kernel")
    wait = body.index("bar(B_PFULL + 2 * sb + h)")
    between = body[body.index("__shfl_sync", wait):body.index("lds_f4(", wait)]
    assert "__syncwarp();" in between


def test_a_give_up_names_its_kernel():
    """Prefill and decode report in the same status word: no two files share the code of a wait."""
    used = {}
    for f in sorted(os.listdir(CSRC)):
        for site in re.findall(r"fail_site = (\d+);|atomicExch\(status \+ 1, (\d+)u\)", open(os.path.join(CSRC, f)).read()):
            used.setdefault(int(site[0] or site[1]), set()).add(f)
    assert used.pop(0) and len(used) > 10 and all(len(files) == 1 for files in used.values()), used
