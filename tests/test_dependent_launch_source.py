"""Kernels that may start before the kernel ahead of them in the stream has
finished (programmatic dependent launch: every kernel that calls
wait_for_previous) must not read what another kernel writes through the
read-only path, nor through a __restrict__ pointer, which the compiler may
load from ahead of the wait.  Checked on the source: the order that a wrong
qualifier loses depends on the build and cannot be provoked in a run."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2311_10314_gb300", "csrc")
# planes formed at create or copied in by the host, written by no kernel of a step
STATIC = {"psi", "psi_pl", "cosf", "inflow"}
# pointers a kernel only stores through, with values formed after the wait
WRITE_ONLY = {("k_step_fused", "pop_out"), ("k_step_fused", "lag_out"), ("k_step_fused", "err"),
              ("k_adj_fields", "mu"), ("k_adj_fields", "chi"),
              ("k_adj_node", "ad_pop_out"), ("k_adj_node", "ad_lag_out"), ("k_adj_gather3", "ad_lag_out")}


def _functions(text):
    """(name, is kernel, parameters, body) of every function template's definition."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"^(__global__|__device__)([^;{]*?)\b(\w+)\(((?:[^(){};]|\([^()]*\))*)\)\s*(?:const\s*)?\{", text, re.M):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(3), m.group(1) == "__global__", m.group(4), text[m.end():i - 1]


def _dependents():
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith(".cu"):
            continue
        fns = list(_functions(open(os.path.join(CSRC, f)).read()))
        helpers = {n: (p, b) for n, k, p, b in fns if not k}
        for n, k, p, b in fns:
            if k and re.search(r"\bwait_for_previous\(\)", b):
                called = [h for h in helpers if re.search(r"\b%s\b" % h, b)]
                yield pytest.param(n, p, b, {h: helpers[h] for h in called}, id="%s:%s" % (f, n))


DEPENDENTS = list(_dependents())


def test_all_dependent_kernels_are_found():
    names = {p.values[0] for p in DEPENDENTS}
    assert names >= {"k_step_fused", "k_open_bc", "k_adj_fields", "k_adj_node", "k_adj_gather3", "k_adj_gather2"}
    text = "".join(open(os.path.join(CSRC, f)).read() for f in os.listdir(CSRC) if f.endswith(".cu"))
    launched = set(re.findall(r"launch_dependent\([^;]*?\b(k_\w+)<", text))
    assert launched == names


@pytest.mark.parametrize("name,params,body,helpers", DEPENDENTS)
def test_dependent_kernels_read_other_kernels_output_by_plain_loads(name, params, body, helpers):
    for const, ptr in re.findall(r"(const\s+)?\w+\s*\*\s*__restrict__\s+(\w+)", params):
        if const:
            assert ptr in STATIC, "%s reads %s through const __restrict__" % (name, ptr)
        else:
            assert (name, ptr) in WRITE_ONLY, "%s: __restrict__ %s" % (name, ptr)
    assert "__ldg" not in body, name
    for h, (hp, hb) in helpers.items():
        assert "__ldg" not in hb, "%s in %s" % (h, name)
        for ptr in re.findall(r"\*\s*__restrict__\s+(\w+)", hp):
            assert ptr in STATIC, "%s: __restrict__ %s of %s" % (name, ptr, h)
