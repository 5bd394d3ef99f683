"""Every device wait has an iteration limit and then returns false, with whatever it waited
for still missing.  These checks read the kernels' sources (an expired wait cannot be
provoked in them): what follows a wait that gave up must not be used as an offset."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2607_27952_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


@pytest.mark.parametrize("name", ["select_gram.cu", "rows_kernels.cu"])
def test_no_wait_result_is_dropped(name):
    src = _source(name)
    assert "mbar_wait_bounded(" in src
    assert re.findall(r"[;{})]\s*mbar_wait_bounded\(", src) == []


def test_workers_read_posted_centres_only_after_a_whole_warp_saw_them():
    """The batch loop of select_gram_kernel: cnt, and through it cen and crow (offsets into the
    matrix), are read only when no lane's wait expired, and a warp leaves the loop together."""
    src = _source("select_gram.cu")
    m = re.search(r"const bool (\w+) = mbar_wait_bounded\(&bars\[i\].*?cnt\[4 \+ i\]", src, re.S)
    assert m, "the wait for a posted batch comes before its count"
    assert re.search(r"if \(!__all_sync\(0xffffffffu, %s\)\) break;" % m.group(1), m.group(0))


@pytest.mark.parametrize("name,kernel,join", [
    ("select_gram.cu", "gram_kernel", "__syncthreads();"),
    ("select_gram.cu", "gram_pair_kernel", "cluster_sync();"),
    ("rows_kernels.cu", "rows_pass_kernel", "__syncthreads();"),
])
def test_copies_in_flight_are_waited_out_whoever_gave_up(name, kernel, join):
    """When any role's wait expires (the issuer's as well as the producer's), copies may still be
    in flight: the CTA waits for them once all roles have joined, before it frees its tensor
    memory and exits."""
    src = _source(name)
    body = src[src.index("%s(const __grid_constant__" % kernel):]
    body = body[:body.index("tmem_dealloc")]
    give = body[body.index("auto twait"):]
    assert "gave_up" in give[:give.index("};")]
    end = body[body.rindex("if (gave_up)") :]
    assert "wait_out(&never)" in end and join in end
    assert body[:body.rindex("if (gave_up)")].rstrip().endswith(join)
