"""Kernels that start early (programmatic dependent launch) and the data they share.

A kernel launched early runs while its predecessor still writes.  __restrict__
and the read-only path promise data that stay the same for a kernel's lifetime,
so only tables that no kernel of an evaluation writes may be read through them;
the states, the staged coefficients and tables and the partials may not.
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_11878_gb300", "csrc")

# Uploaded or built when a plan or a Hamiltonian is set, before any evaluation.
PLAN_TABLES = {"groups", "tz", "tc", "hdiag", "wgroups", "wterms", "hoff", "gates", "desc", "order", "pat",
               "ca", "cb", "off", "count", "step"}


def _early_kernels():
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for part in text.split("__global__")[1:]:
            body = part[: part.index("\n}")]
            if "pdl_wait()" not in body:
                continue
            head = body[: body.index("{")]
            name = re.findall(r"\b(k_\w+)\s*\(", head)[0]
            found.append((os.path.basename(path), name, head[head.index(name) + len(name):]))
    return found


def test_the_early_kernels_are_found():
    names = {k[1] for k in _early_kernels()}
    assert names == {"k_energy_cols", "k_apply_h", "k_energy_finish", "k_grad_finish", "k_energy_win",
                     "k_apply_h_win", "k_exc_pass", "k_pass", "k_pass_fixed", "k_pass_fx", "k_apply_h_sweep"}


@pytest.mark.parametrize("kernel", _early_kernels(), ids=lambda k: k[1])
def test_restrict_only_on_plan_tables(kernel):
    assert set(re.findall(r"__restrict__\s+(\w+)", kernel[2])) <= PLAN_TABLES


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_read_only_loads_only_from_plan_tables(path):
    text = re.sub(r"//[^\n]*", "", open(path).read())
    if "k_build_hdiag" in text:    # launched plainly, its c and z are terms of H
        text = re.sub(r"k_build_hdiag.*?\n}", "", text, count=1, flags=re.S)
    assert set(re.findall(r"__ldg\(\s*(\w+)", text)) <= PLAN_TABLES
