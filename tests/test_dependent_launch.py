"""What the kernels may touch before they wait for the kernel before them
(programmatic dependent launch), checked on the sources: a mistake here is a
race that a run shows rarely or never, so no run is asked to show it."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2111_09294_gb300", "csrc")


def functions():
    """(file, name, parameters, body) of every function, comments removed."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = re.sub(r"/\*.*?\*/|//[^\n]*", "", open(path).read(), flags=re.S)
        for m in re.finditer(r"^(?:__global__|__device__|template|static|inline|void)[^;{}]*?"
                             r"(\w+)\(((?:[^(){};]|\([^(){};]*\))*)\)\s*(?:const\s*)?\{",
                             src, flags=re.M):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
            yield os.path.basename(path), m.group(1), m.group(2), src[m.end():i - 1]


def before_wait():
    """(file, name, text before the first wait) of the functions that wait."""
    return [(f, n, b[:b.index("pdl_wait()")]) for f, n, _, b in functions() if "pdl_wait()" in b]


def test_every_waiting_kernel_is_found():
    names = {n for _, n, _ in before_wait()}
    assert {"k_spmv", "k_spmv_lean", "spmm_body", "k_update", "k_restrict", "prolong_box",
            "restrict_update_unit", "prolong_rows_unit", "k_coarse", "k_coarse32",
            "restrict_b_unit", "coarse_b_body", "prolong_b_unit", "k_block_apply",
            "k_renumber"} <= names


# the run's scalars change while kernels run: before the wait they are read from
# L2 only, and only to decide whether to start loading
@pytest.mark.parametrize("where", before_wait(), ids=lambda w: f"{w[0]}:{w[1]}")
def test_scalars_before_the_wait_come_from_l2(where):
    plain = re.sub(r"(?:ld_early|__ldcg)\(&(?:bs|sc)->\w+\)", "", where[2])
    assert not re.search(r"\b(?:bs|sc)->", plain), where[:2]


def test_a_held_system_is_not_read_before_the_wait():
    # in a launch over several systems a replacement may be writing the system's
    # vectors and scalars: nothing but the tables and Z~ before the wait
    text, = [t for _, n, t in before_wait() if n == "prolong_b_unit"]
    assert not re.search(r"\ba\.(?:p|rA|rB|NU32)\b|&?bs->", text)


# vectors that an earlier kernel of the run wrote are complete before some waits,
# but visible to ordinary loads only after them: from L2 there (a thread's own
# arrays have an index of their own, i, or a size)
@pytest.mark.parametrize("where", before_wait(), ids=lambda w: f"{w[0]}:{w[1]}")
def test_vectors_before_the_wait_come_from_l2(where):
    plain = re.findall(r"(?:(?<![.\w])|\ba\.)(?:r_cur|yv|y|p|u|q|r|x|a|b)\[([^\]]*)\]", where[2])
    # (prolong_box's lambda of such loads is called after the wait only)
    own = {"i", "R", "3"} | ({"d + i"} if where[1] == "prolong_box" else set())
    assert not set(plain) - own and not re.search(r"^\s*load3\(", where[2], re.M), where[:2]


# set-up data, complete before any kernel of a run: the tables and their offsets,
# E^-1, the restriction's records and its blocks of W
SETUP = {"off", "off + mid", "off + s", "off + s + 1", "tab", "Einv", "r2 + j", "r2 + j + 32",
         "row + j", "row + j + 32", "B.ext.rec + e0 + ch0 * CE + i",
         "B.own.rec + z0 + ch0 * CO + i", "b + i * M"}


def test_read_only_loads_are_of_setup_data():
    waiting = {n for _, n, _ in before_wait()} | {"k_spmm_sys", "k_restrict_b_sys", "load",
                                                  "k_coarse_b_sys", "k_prolong_b_sys", "sys_of"}
    for f, n, params, body in functions():
        for arg in re.findall(r"__ldg\(((?:[^()]|\([^()]*\))*)\)", body):
            assert arg in SETUP, (f, n, arg)
        if n in waiting:
            # what is only written (y) may be told apart from the rest
            for const, name in re.findall(r"(const )?[\w<>]+ \*__restrict__ (\w+)", params + body):
                assert not const or name in SETUP, (f, n, name)


def test_tiles_beside_another_kernel_are_read_from_l2():
    # the dense inverse's trailing update runs beside a kernel without waiting
    # for it before it works: no ordinary load of the matrix or the panel
    body, = [b for _, n, _, b in functions() if n == "update_tile"]
    loads = re.sub(r"ld_early\((?:[^()]|\((?:[^()]|\([^()]*\))*\))*\)", "L2", body)
    assert "mat_at" not in re.sub(r"\*mat_at\([^()]*\) = |double \*t = mat_at\([^()]*\);", "", loads)
    assert not re.search(r"\bC\[|-=", loads)
    assert re.findall(r"\*t\b[^;]*;", re.sub(r"double \*t = [^;]*;", "", loads)) == [
        "*t = L2 - X[ii * kLd + jj];"]
