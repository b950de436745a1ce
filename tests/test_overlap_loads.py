"""Kernels that may start while their predecessor still writes (programmatic
dependent launch) read the vectors with plain loads after their wait: no
__restrict__ on a vector parameter, which would let the compiler move its loads
above the wait or send them through the read-only path, and no explicit
read-only load of one.  Checked in the source, without a GPU."""

import os
import re

import pytest

SRC = os.path.join(os.path.dirname(__file__), "..", "paper_1506_06185_gb300", "csrc", "kernels.cu")
# parameters that hold what the host wrote at set-up
TABLES = set("rs rsf rsc W Winv Wv Wsc winv tiles act cptr cps cpo list items slots gather zero_off if_gid gid geo "
             "rowptr col val fsrc uptr udst umaster dinv idx ids off master".split())
# position of the "read-only path" argument in the template arguments of the
# functions that load vectors (a ZERO residual, argument 3, loads nothing)
NC_ARG = {"gs_group7": 2, "gs_group15": 1, "gs_tile7": 2, "res_group7": 4, "res_group15": 4, "restrict_slot": 1,
          "restrict_tile": 1, "prolong_slot": 1, "prolong_group": 1, "prolong_tile": 1}


def _closing(s, at, pair):
    depth = 0
    for q in range(at, len(s)):
        depth += (s[q] == pair[0]) - (s[q] == pair[1])
        if depth == 0:
            return q
    raise ValueError("unbalanced")


def waiting_functions(src):
    """name -> (parameters, body) of every kernel that waits for its
    predecessor, and of the functions that wait for them."""
    src = re.sub(r"//[^\n]*", "", src)
    found = {}
    for m in re.finditer(r"(?:__global__|__device__)[^;{}()]*(?:__launch_bounds__\([^{};]*?\)\s*)?\b(\w+)\((?=[^()]*\b)", src):
        if m.group(1) == "__launch_bounds__":
            continue
        end = _closing(src, m.end() - 1, "()")
        brace = src.find("{", end)
        if brace < 0 or src[end + 1:brace].strip():
            continue
        body = src[brace:_closing(src, brace, "{}") + 1]
        found[m.group(1)] = (src[m.end():end], body, "__global__" in m.group(0))
    waits = {n for n, (_, b, _) in found.items() if "after_previous()" in b and n != "after_previous"}
    return {n: found[n][:2] for n in found
            if n in waits or (found[n][2] and any(re.search(r"\b%s\b" % w, found[n][1]) for w in waits))}


FUNCS = waiting_functions(open(SRC).read())


def test_found_the_kernels():
    for name in ("k_gs", "k_gs_flat", "gs_if_prefetched", "k_res", "k_res_flat", "k_restrict", "k_restrict_flat",
                 "k_prolong", "k_prolong_flat", "k_gs_stream", "k_res_f32", "k_add_corr_blocks", "k_cg",
                 "k_cg_cluster", "k_reduce", "k_import", "k_export", "k_restore", "k_zero_blocks"):
        assert name in FUNCS, name


@pytest.mark.parametrize("name", sorted(FUNCS))
def test_vectors_are_read_with_plain_loads(name):
    params, body = FUNCS[name]
    restricted = {p.split()[-1].lstrip("*&") for p in re.split(r",(?![^<]*>)", params) if "__restrict__" in p}
    assert restricted <= TABLES, sorted(restricted - TABLES)
    for arg in re.findall(r"__ldg\(\s*(?:A\.)?(\w+)", body):
        assert arg in TABLES, arg
    for m in re.finditer(r"\b(%s)<([^<>()]*)>\(" % "|".join(NC_ARG), body):
        args = [a.strip() for a in m.group(2).split(",")]
        if m.group(1).startswith("res_group") and len(args) == 4 and args[3] == "true":
            continue
        at = NC_ARG[m.group(1)]
        assert len(args) > at and args[at] in ("!DEP", "false"), m.group(0)
