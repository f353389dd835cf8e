"""Kernels launched while their predecessor still runs read its results only after the wait (checked in the sources).

Such a kernel (launch_pdl, launch_pdl_ex) may start before the kernel in front of it has finished. What the chain of
launches writes is read through a pointer that the compiler learns at or after the wait (pdl_wait, relearn), or by a
volatile load (__ldca, __ldcg, __ldcs, load_after_wait, gate_closed, atomics): the compiler may move any other load above the
wait. Every pointer that a kernel gets is classified here, so that a new kernel or parameter has to be looked at:

  const    constant over the chain: operators, tables, coefficients
  plain    not __restrict__: the wait's memory clobber orders its loads
  learned  named in pdl_wait() or relearn(), as it is or as the pointer formed from it
  volatile loaded only by the volatile forms, and otherwise only written
  formed   pointers formed from the others (or from the tables) that are named in relearn()
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1701_03989_gb300", "csrc")

KERNELS = {
    "mpk_items_kernel": dict(const="descs items", volatile="sys_steps emax_all", formed="x"),
    "mpk_items_both_kernel": dict(const="descs items", volatile="sys_steps"),
    "recover_items_kernel": dict(const="descs items", volatile="sys_w coords"),
    "gram_partial_kernel": dict(volatile="Y partials gate"),
    "gram_items_kernel": dict(const="descs items", volatile="sys_w partials"),
    "gram_items_moment_finalize_kernel": dict(const="sys_item0 sys_nitems", learned="partials", volatile="sys_w G"),
    "gram_finalize_kernel": dict(learned="partials", volatile="G gate"),
    "gram_items_finalize_kernel": dict(const="sys_item0 sys_nitems", learned="partials", volatile="sys_w G"),
    "mpk_split_step_kernel": dict(plain="Y emax_part", volatile="oval dtil gate"),
    "mpk_chain_step_kernel": dict(plain="emax_part", volatile="oval dtil Y gate", formed="v x"),
    "emax_reduce_kernel": dict(volatile="emax_part col_emax gate"),
    "recover_kernel": dict(learned="coords", plain="Y x r p", volatile="gate"),
    "cg_spmv_dot_kernel": dict(plain="p st partials counter", volatile="q"),
    "cg_update_kernel": dict(plain="st partials counter res_hist alpha_hist beta_hist", volatile="r q"),
    "cg_pupdate_kernel": dict(plain="st", volatile="x r p"),
    "block_ctrl_kernel": dict(const="th_g sg_g gm_g", learned="G", plain="st counters", volatile="coords hist res_hist ab_hist spec"),
    "block_handover_kernel": dict(plain="prev host_rec host_seq cur"),
    # the two flags and sys_w were written several kernels before and are read ahead of the wait
    "gram_tc_kernel": dict(volatile="col_emax partials"),
    "gram_tc_items_kernel": dict(const="pieces sys_w", volatile="emax_all partials sums tickets"),
    "recover_tc_kernel": dict(learned="x", plain="failed", volatile="col_emax coords r p"),
}


def _code(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


def _sources():
    return {f: _code(f) for f in sorted(glob.glob(os.path.join(CSRC, "*.cu")))}


def _balanced(text, i, pair):
    depth = 0
    for k in range(i, len(text)):
        depth += (text[k] == pair[0]) - (text[k] == pair[1])
        if depth == 0:
            return k
    raise AssertionError("unbalanced")


def _kernel(name):
    """Parameter list and body of a __global__ function."""
    for text in _sources().values():
        for m in re.finditer(r"__global__\s+void\s+[^;{]*?\b%s\s*\(" % name, text):
            e = _balanced(text, m.end() - 1, "()")
            b = text.index("{", e)
            return text[m.end(): e], text[b: _balanced(text, b, "{}") + 1]
    raise AssertionError(name)


def _pointers(params):
    return set(re.findall(r"\*\s*(?:__restrict__\s+)?(\w+)\s*(?:,|$)", params))


def _launched():
    names = set()
    for text in _sources().values():
        names |= set(re.findall(r"launch_pdl(?:_ex)?\(\s*(\w+)", text))
    return names


def test_every_dependent_kernel_is_listed():
    assert _launched() == set(KERNELS)


@pytest.mark.parametrize("name", sorted(KERNELS))
def test_reads_after_the_wait(name):
    params, body = _kernel(name)
    spec = {k: set(v.split()) for k, v in KERNELS[name].items()}
    const, plain, learned, vol = (spec.get(k, set()) for k in ("const", "plain", "learned", "volatile"))
    assert _pointers(params) == const | plain | learned | vol, "every pointer parameter is classified"
    for p in plain:
        assert not re.search(r"__restrict__\s+%s\b" % p, params), p
    taken = set(re.findall(r"\w+", " ".join(re.findall(r"(?:pdl_wait|relearn)\(([^)]*)\)", body))))
    assert learned | spec.get("formed", set()) <= taken
    for p in vol:  # no ordinary load: written, handed on, or inside a volatile form
        rest = re.sub(r"(?:__ldcg|__ldcs|__ldca|load_after_wait|gate_closed|atomic\w+)\((?:[^()]|\([^()]*\))*\)", "", body)
        for m in re.finditer(r"(?<![\w.>])%s\s*\[" % p, rest):
            after = rest[_balanced(rest, m.end() - 1, "[]") + 1:].lstrip()
            assert re.match(r"=(?!=)", after), (p, rest[m.start(): m.start() + 60])
        assert not re.search(r"__ldg\(\s*%s\b" % p, rest), p
    assert not re.search(r"__ldg\(\s*(?:[pr]j|cq|d\.Y|d\.x)\b", body)
    for p in taken:  # what is learned after the wait may be written during the chain
        assert not re.search(r"__ldg\(\s*%s\s*[+)]" % p, body) or p == "v", p
    assert "pdl_wait(" in body or "gram_tc_body(" in body


def test_row_sums_gather_by_ordinary_loads():
    """x of the row sums is the previous kernel's result."""
    text = _code(os.path.join(CSRC, "ascg_common.cuh")) + _code(os.path.join(CSRC, "kernels_cg.cu"))
    assert not re.search(r"__ldg\(\s*x\b", text)
