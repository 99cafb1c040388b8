"""Rules of the device code that a run does not show when they are broken (what follows is undefined
rather than wrong each time), checked on the sources."""

import glob
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_30738_gb300", "csrc")
KERNELS = sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _code(path):
    """The file's text with its comments and strings blanked out."""
    text = open(path).read()
    return re.sub(r'//[^\n]*|/\*.*?\*/|"(?:\\.|[^"\\\n])*"', lambda m: re.sub(r"[^\n]", " ", m.group()), text,
                  flags=re.S)


def _function(code, name):
    """Text of the body of function `name`."""
    at = re.search(r"\b%s\s*\([^;{]*\)\s*\{" % name, code).end()
    depth, end = 1, at
    while depth:
        depth += {"{": 1, "}": -1}.get(code[end], 0)
        end += 1
    return code[at:end - 1]


def _headers(code, at):
    """What stands before each block that is open at position `at`, and the statement up to it."""
    open_at, depth = [], 0
    for i in range(at - 1, -1, -1):
        if code[i] == "}":
            depth += 1
        elif code[i] == "{":
            if depth:
                depth -= 1
            else:
                open_at.append(i)
    starts = [at] + open_at
    return [re.split(r"[;{}]", code[:i])[-1] for i in starts]


@pytest.mark.parametrize("path", KERNELS, ids=os.path.basename)
def test_whole_warps_wait_together(path):
    # the lanes of a warp may leave a bounded wait at different times: code that a whole warp runs
    # waits by warp_wait, which brings them together again for the aligned instructions behind it
    code = _code(path)
    for m in re.finditer(r"\bmbar_wait2?\(", code):
        one = r"(lane|threadIdx\.x|tid)\s*==\s*0"
        assert any(re.search(one, h) for h in _headers(code, m.start())), code[:m.start()].count("\n") + 1


def test_greedy_has_no_branch_between_tmem_load_and_wait():
    body = _function(_code(os.path.join(CSRC, "kve_select.cu")), "gram_greedy")
    between = re.search(r"tmem_ld1\((.*?)tmem_wait_ld\(", body, flags=re.S).group(1)
    assert not re.search(r"\b(if|for|while)\b", between)


@pytest.mark.parametrize("path", KERNELS, ids=os.path.basename)
def test_tmem_waits_name_what_was_loaded(path):
    # a wait that does not name the loaded registers does not keep their readers behind it
    waited = re.findall(r"\btmem_wait_ld\(([^()]*)\)", _code(path))
    loaded = re.findall(r"\btmem_ld\w+\(", _code(path))
    assert bool(waited) == bool(loaded) and all(w.strip() for w in waited)
    assert not re.search(r"tmem_wait_ld\(\s*\)", _code(os.path.join(CSRC, "kve_ptx.cuh")))


def test_select_reads_keys_inside_the_unit():
    # wherever a pool position becomes a key's address, it has been checked
    body = _function(_code(os.path.join(CSRC, "kve_select.cu")), "select_kernel")
    at = [m.start() for m in re.finditer(r"P\.k \+", body)]
    assert len(at) == 2
    assert all(any("pos >= 0 && pos < Lc" in h for h in _headers(body, i)) for i in at)


@pytest.mark.parametrize("path", KERNELS, ids=os.path.basename)
def test_dependent_launches_take_no_tmem_early(path):
    # a kernel that may start while its predecessor runs holds no TMEM before that has finished: the
    # predecessor can be a caller's kernel that still has to allocate its own
    code = _code(path)
    for name in set(re.findall(r"\b(\w+_kernel)\s*\(const", code)):
        body = _function(code, name)
        if "wait_previous_kernel(" in body and "tmem_alloc(" in body:
            assert body.index("wait_previous_kernel(") < body.index("tmem_alloc("), name
    if os.path.basename(path) == "kve_select.cu":
        assert "tmem_alloc(" in _function(code, "select_kernel")


def test_select_decodes_only_what_the_greedy_wrote():
    # after a wait that ran out no admission was written: the unit leaves before its tie keys, which
    # index the pool, are decoded
    body = _function(_code(os.path.join(CSRC, "kve_select.cu")), "select_kernel")
    at = body.index("gram_greedy<NT>(")
    assert at < body.index("if (!formed)", at) < body.index("adm_slot[t]", at)
