"""Rules that the CUDA sources keep where kernels of a stream overlap (programmatic dependent
launch) or run instructions that want a converged warp, checked on the source text: what breaks
them compiles, and may well give the right results on the machine at hand."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2609_35593_gb300", "csrc")


def _code(path):
    """The file without its comments."""
    text = re.sub(r"/\*.*?\*/", " ", open(path).read(), flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def _balanced(text, at, pair):
    """text[at:] up to the bracket that closes the one at `at`."""
    depth = 0
    for k in range(at, len(text)):
        depth += (text[k] == pair[0]) - (text[k] == pair[1])
        if depth == 0:
            return text[at:k + 1]
    raise AssertionError("unbalanced")


def _kernels():
    """(name, parameter list, body) of every kernel."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = _code(path)
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\s*)?", text):
            at = m.end()
            if text[at] == "(":
                at += len(_balanced(text, at, "()"))
            name = re.compile(r"\s*(\w+)\s*").match(text, at)
            params = _balanced(text, name.end(), "()")
            body = _balanced(text, text.index("{", name.end() + len(params)), "{}")
            out.append((name.group(1), params, body))
    return out


OVERLAPPED = [k for k in _kernels() if "pdl_wait" in k[2]]


def test_the_overlapped_kernels_are_found():
    names = {k[0] for k in OVERLAPPED}
    assert {"k_pool", "k_zproj", "k_dot", "k_dot_run", "k_yagg", "k_score_rows", "k_round_rows",
            "k_pairing", "k_rowptr", "k_csr", "k_pairs", "k_attn", "k_oproj"} == names


@pytest.mark.parametrize("name,params", [k[:2] for k in OVERLAPPED], ids=[k[0] for k in OVERLAPPED])
def test_overlapped_kernels_promise_nothing_about_aliasing(name, params):
    # the kernel ahead may still write what such a parameter points to
    assert "__restrict__" not in params, name


def test_no_read_only_loads():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        assert not re.search(r"ld\.global\.nc|__ldg\b|\.nc\.", _code(path)), path
