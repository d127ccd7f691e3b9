"""Host check of the sources: what a step kernel reads while another grid may
still write it (populations, the beta-stencil's c) is not
read through the read-only path.  The step kernels and the products may start
before the kernel ahead of them in the stream has ended (griddepcontrol), so
that memory is not constant for their lifetime, and a load declared invariant
is not ordered behind griddepcontrol.wait.  A race has no certain outcome to
run against, so the rule is checked where it is kept."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_10399_gb300", "csrc")
READ_ONLY = re.compile(r"__ldg|ld\.global(\.\w+)*\.nc|__builtin_nontemporal_load|__restrict__")


def _source(name):
    s = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", s, flags=re.S)


def _bodies(src, name):
    """Parameter lists and bodies of the definitions of function `name`."""
    out = []
    for m in re.finditer(r"\b%s\(" % name, src):
        i = src.index(")", m.end())
        j = re.compile(r"[{;]").search(src, i).start()
        if src[j] == ";" or not re.match(r"\)[\s\w]*$", src[i:j]):
            continue  # a call
        depth, k = 1, j + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(src[k], 0)
            k += 1
        out.append(src[m.start():k])
    return out


@pytest.mark.parametrize("name, count", [("ld_raw", 2), ("load_c", 1), ("stage_c_halo", 1), ("load_beta", 1),
                                         ("fused_step_node", 1)])
def test_step_reads_are_ordinary_loads(name, count):
    got = _bodies(_source("lbm_kernels.cuh"), name)
    assert len(got) == count, name
    for b in got:
        assert not READ_ONLY.search(b), b[:200]


def test_node_loads_are_ordinary_loads():
    src = _source("lbm_kernels.cuh")
    at = src.index("void load_node(")
    body = src[at:src.index("struct Moments", at)]
    assert "pop_offset" in body and not READ_ONLY.search(body)


@pytest.mark.parametrize("name", ["lbm_pairs.cuh", "lbm_ref_1d.cuh"])
def test_files_without_read_only_loads(name):
    assert not READ_ONLY.search(_source(name))


def test_products_read_only_the_bias_that_way():
    """Parameters are not written by a kernel that a product can overlap with:
    the optimiser's is followed by kernels launched in full order."""
    src = _source("fno_umma.cuh")
    assert len(READ_ONLY.findall(src)) == src.count("__ldg(g.bias ") == 2
    fno = _source("lbm_fno.cu")
    adam = fno.index("k_adam<<<")
    assert "refresh_weights(f)" in fno[adam:adam + 600]
    (body,) = _bodies(_source("fno_kernels.cuh"), "k_adam")
    assert "let_next_start" not in body


def test_the_batch_reads_only_its_constant_tables_early():
    """k_batch_step may read its argument table and work list before it waits:
    no kernel writes them."""
    src = _source("lbm_kernels.cuh")
    at = src.index("k_batch_step(")
    body = src[at:src.index("fused_step_node", at)]
    wait = body.index("wait_previous")
    assert [m.group(0) for m in READ_ONLY.finditer(body)] == ["__restrict__", "__restrict__", "__ldg"]
    assert "a.pop" not in body[:wait] and not READ_ONLY.search(body[wait:])


def test_a_step_lets_the_next_go_after_its_own_wait():
    """Let go before the wait, the blocks of several steps to come would hold
    the SMs that a step of few blocks needs."""
    (body,) = _bodies(_source("lbm_kernels.cuh"), "wait_previous")
    assert 0 < body.index("griddepcontrol.wait") < body.index("griddepcontrol.launch_dependents")
