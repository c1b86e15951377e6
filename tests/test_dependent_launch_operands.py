"""Operands of the kernels that start under their predecessor (dep_begin / dep_wait): a `const
__restrict__` operand promises data unchanged over the kernel's whole lifetime, which only tables made at
plan or batch creation are. Read from the sources; needs no GPU."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2307_00391_gb300", "csrc")

# made at plan or batch creation and never written again
TABLES = {
    "k_clock_block": {"rot"},
    "k_clock_spec": {"rot", "ph_lo", "ph_hi", "roots"},
    "k_toeplitz_rows": {"g"},
    "k_toeplitz_rows_ks": {"g"},
    "k_spec_rows": {"B"},
    "k_spec_matvec": {"B"},
    "k_spec_tree": {"frac", "rot"},
}


def _close(s, i, pair):
    depth = 0
    for j in range(i, len(s)):
        depth += (s[j] == pair[0]) - (s[j] == pair[1])
        if depth == 0:
            return j
    raise ValueError("unbalanced")


def _functions(src):
    """(name, qualifier, parameters, body) of the device code of one source file."""
    src = re.sub(r"//[^\n]*", "", src)
    src = re.sub(r"__launch_bounds__\((?:[^()]|\((?:[^()]|\([^()]*\))*\))*\)", "", src)
    for m in re.finditer(r"__(global|device)__[^;{}()]*?\b(\w+)\(", src):
        end = _close(src, m.end() - 1, "()")
        if not re.match(r"\s*\{", src[end + 1:]):
            continue
        body = src.index("{", end)
        yield m.group(2), m.group(1), src[m.end():end], src[body:_close(src, body, "{}")]


def _read_only(params):
    return set(re.findall(r"const [\w:<> ]+\*\s*__restrict__ (\w+)", params))


@pytest.fixture(scope="module")
def functions():
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        out += list(_functions(open(path).read()))
    return out


def test_only_tables_are_read_only(functions):
    kernels = {n: (p, b) for n, q, p, b in functions if q == "global" and re.search(r"\bdep_(begin|wait)\(\)", b)}
    assert len(kernels) >= 27 and set(TABLES) <= set(kernels)
    found = {n: _read_only(p) for n, (p, _) in kernels.items() if _read_only(p)}
    assert found == TABLES


def test_their_helpers_take_the_state_plainly(functions):
    helpers = {n: p for n, q, p, _ in functions if q == "device" and n.startswith("measure_")}
    assert len(helpers) >= 4
    assert not any(_read_only(p) for p in helpers.values())


def test_every_dependent_launch_waits(functions):
    """Every kernel launched with launch_dep or the attribute itself calls dep_begin or dep_wait."""
    waits = {n for n, q, _, b in functions if q == "global" and re.search(r"\bdep_(begin|wait)\(\)", b)}
    launched = set()
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        launched |= set(re.findall(r"launch_dep\((k_\w+)", open(path).read()))
    assert launched and launched <= waits, launched - waits
