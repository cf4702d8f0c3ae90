"""Order of the kernels launched while their predecessor still runs
(launch_dependent in csrc/common.cuh): before such a kernel executes
grid_dep_wait() it may read only what was written two or more kernels
earlier.  Every pointer that a kernel's source names before its first wait is
compared with the list of those that are safe there, each with its writer.
A misplaced read is a race, so it is looked for in the source."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2609_06086_gb300", "csrc")
TEXT = {os.path.basename(f): re.sub(r"//[^\n]*", "", open(f).read())
        for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*")))}

# kernel -> pointers it may read before any wait, and who writes them
TABLES = "cost tables: the handle's set-up, or the search's first kernel (a search's later " \
         "kernels have waited for it, each for the one before)"
EARLY = {
    "bound_kernel": {"blob": TABLES},
    "level_kernel": {"p.blob": TABLES},
    "leaf_kernel": {"p.blob": TABLES},
    "decode_kernel": {"p.blob": TABLES},
    "eval_kernel": {"p.tblob": TABLES, "p.offs": "sort_scatter_kernel; decode_kernel is between"},
    "short_kernel": {"p.tblob": TABLES, "p.offs": "sort_scatter_kernel; decode_kernel is between"},
    "il_eval_kernel": {"p.cblob": TABLES},
}
# kernels with a first wait under a condition: the condition, and what is safe
# between it and the wait of every instance
LATER = {
    "level_kernel": ("if constexpr (X == 0)",
                     {"p.slices": "gather_kernel; at depths above 0 a level kernel is between",
                      "p.vb": "bound_kernel; gather_kernel is between"}),
    "il_eval_kernel": ("if (p.offs_last)",
                       {"p.offs": "sort_scatter_kernel, decode_kernel between; offs_last is set "
                                  "where il_offs_kernel writes them right before"}),
}


def braces(text, at):
    """The text between the brace at or after `at` and its partner."""
    i = text.index("{", at)
    depth, j = 0, i
    while True:
        depth += (text[j] == "{") - (text[j] == "}")
        if depth == 0:
            return text[i + 1:j]
        j += 1


def kernels():
    """(name, parameter list, body) of every kernel that waits for another."""
    out = []
    for text in TEXT.values():
        for m in re.finditer(r"__global__[\w\s(),<>:]*?\b(\w+)\s*\(((?:[^()])*)\)\s*\{", text):
            body = braces(text, m.end() - 1)
            if "grid_dep_wait()" in body:
                out.append((m.group(1), m.group(2), body))
    return out


def pointers(params):
    """Pointer parameters, and p.<member> for the pointer members of a
    parameter struct."""
    names = set(re.findall(r"\*\s*(\w+)", params))
    for struct in re.findall(r"\b(\w+Params)\s+p\b", params):
        for text in TEXT.values():
            m = re.search(r"\bstruct %s\s*\{" % struct, text)
            if m:
                for decl in re.findall(r"([^;{}]*\*[^;{}]*);", braces(text, m.end() - 1)):
                    names |= {"p." + n for n in re.findall(r"\*\s*(\w+)", decl)}
                    names |= {"p." + n for n in re.findall(r",\s*(\w+)", decl)}
    assert names
    return names


def read_in(part, names):
    return {n for n in names if re.search(r"(?<![\w.])%s\b" % re.escape(n), part)}


KERNELS = kernels()


def test_the_kernels_are_found():
    names = {k[0] for k in KERNELS}
    assert {"feas_kernel", "lim_kernel", "sort_scatter_kernel", "argmin_final"} <= names
    assert set(EARLY) <= names


@pytest.mark.parametrize("kernel", KERNELS, ids=[k[0] for k in KERNELS])
def test_reads_before_the_wait(kernel):
    name, params, body = kernel
    names = pointers(params)
    # a wait on the way out of a block without work orders none of its reads
    parts = re.sub(r"grid_dep_wait\(\);\s*return;", "return;", body).split("grid_dep_wait()")
    counters = {"stats", "p.stats"}  # raised when the tables' staging ran out of polls
    early = read_in(parts[0], names) - counters
    assert early <= set(EARLY.get(name, {})), early - set(EARLY.get(name, {}))
    if name in LATER:
        cond, safe = LATER[name]
        assert re.sub(r"\s+", " ", parts[0]).rstrip().endswith(cond)
        between = read_in(parts[1], names) - counters
        assert between <= set(safe) | set(EARLY[name]), between
