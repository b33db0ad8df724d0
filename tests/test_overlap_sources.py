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


def _helpers():
    """(file:name, body) of every device function with an instruction that is .aligned over the
    warp besides TMEM loads and stores (bar.* without .cta is short for barrier.cta.aligned)."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = _code(path)
        for m in re.finditer(r"__device__ __forceinline__ [\w ]+?\b(\w+)\(", text):
            params = _balanced(text, m.end() - 1, "()")
            body = _balanced(text, text.index("{", m.end() - 1 + len(params)), "{}")
            if re.search(r'barrier\.cluster|"bar\.|tcgen05\.(?:de)?alloc', body):
                out.append((m.group(1), body))
    return out


HELPERS = _helpers()


def test_the_aligned_helpers_are_found():
    assert sorted(k[0] for k in HELPERS) == sorted(
        ["tmem_alloc", "tmem_dealloc", "tmem_alloc_pair", "tmem_dealloc_pair", "cluster_sync", "conv_sync",
         "o_epi_sync", "o_epi_sync_all", "o_epi_sync_and", "o_epi_sync_and_all"])


@pytest.mark.parametrize("name,body", HELPERS, ids=[k[0] for k in HELPERS])
def test_aligned_helpers_converge_the_warp_first(name, body):
    first = body.find("__syncwarp()")
    assert 0 <= first < body.index("asm"), name


def test_product_tiles_converge_the_warp_before_they_read_tmem():
    # one lane hands each box of 32 columns to a bulk store and is back at the next box's load
    text = _code(os.path.join(CSRC, "k_dot.cu"))
    loads = list(re.finditer(r"RESS_TMEM_LD32", text))
    assert len(loads) == 2
    for m in loads:
        assert text[:m.start()].rstrip().endswith("__syncwarp();")
