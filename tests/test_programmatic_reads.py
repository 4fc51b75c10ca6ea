"""Kernels launched while the one before still runs (launch_next): what another kernel of the
chain writes is read only through fresh(), after the wait, and by coherent loads.  A race that a
compiler may or may not make of a const __restrict__ read cannot be provoked, so the sources are
read: every kernel of a chain, the arrays it takes from the others, and every __ldg left."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2111_06704_gb300", "csrc")

# kernel: the arrays another kernel of its chain may have written
TAKES = {
    "pcg.cu": {
        "k_matvec_f64": ["pv", "st"],
        "k_matvec_f32": ["pv", "plo", "p64", "st"],
        "k_matvec_stream": ["a.xt", "a.p64", "a.st"],
        "k_matvec_ragged": ["pv", "plo", "p64", "st"],
        "k_update": ["st", "x", "r", "z", "p", "q", "pq_part"],
        "k_dc_apply": ["st", "r", "z", "dots"],
        "k_dc_apply_ordered": ["st", "r", "z", "dots"],
        "k_dc_apply_t": ["st", "rt", "r", "z", "rsum_part"],
        "k_step": ["a.dots", "a.rz.p", "a.cur", "z", "p"],
    },
    "potential.cu": {
        "k_axis_phasors": ["sfix"],
        "k_ion_sf_f64": ["axis"],
        "k_ion_sf_f32": ["sion"],
        "k_bsol_kspace_f64": ["v"],
        "k_bsol_kspace_f32": ["v", "vhead", "bsol"],
    },
    "real_space.cu": {
        "k_bsol_real": ["a.ions"],
        "k_bsol_finish": ["a.part", "a.sums", "a.bsol_k", "a.far", "a.far_state", "a.far_row",
                          "a.far_count"],
    },
    "forces.cu": {
        "k_force_kspace": ["sion", "v", "vhead"],
        "k_force_kspace_f64": ["axis", "v"],
        "k_force_real": ["sion"],
        "k_force_finish": ["kpart", "rpart", "slab"],
    },
}

# what __ldg may read: the matrix and its rows, P's pattern and entries, the tables, the operand
LDG = {"pcg.cu": {"e", "idx", "prow"}, "potential.cu": {"turn", "a", "p", "Ahead"},
       "real_space.cu": {"T"}, "forces.cu": set(), "phasor.cuh": {"T"}}


def _text(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _kernel(text, name):
    """The kernel's body: from its opening brace to the first closing one in column 0."""
    at = re.search(r"^%s\(|\s%s\((?=[^;]*\)\s*\{)" % (name, name), text, re.M).start()
    return text[text.index("{\n", at):text.index("\n}\n", at)]


@pytest.mark.parametrize("name", sorted(TAKES))
def test_every_kernel_of_a_chain_is_listed(name):
    launched = set(re.findall(r"launch_next\(\s*(?:\w+\s*\?\s*)?(k_\w+)", _text(name)))
    launched |= set(re.findall(r":\s*(k_\w+)<[^>]*>,\s*(?:dim3|gv)", _text(name)))
    kernels = {k for k in launched if k.startswith("k_")}
    assert kernels <= set(TAKES[name])
    waiting = set()
    for k in re.findall(r"(k_\w+)\(", _text(name)):
        if re.search(r"\b%s\([^;{]*\)\s*\{" % k, _text(name)) and \
                "wait_previous(" in _kernel(_text(name), k):
            waiting.add(k)
    assert waiting == set(TAKES[name])


@pytest.mark.parametrize("name,kernel", [(f, k) for f in TAKES for k in TAKES[f]])
def test_reads_come_after_the_wait(name, kernel):
    body = _kernel(_text(name), kernel)
    wait = body.index("wait_previous(")
    for array in TAKES[name][kernel]:
        at = body.find("fresh(%s)" % array)
        assert at > wait, (kernel, array)
        if "." not in array:  # the parameter itself is replaced, and not used before
            assert re.search(r"\b%s = fresh\(%s\)" % (array, array), body), (kernel, array)
            assert not re.search(r"\b%s\s*[\[+]" % array, body[:at]), (kernel, array)


@pytest.mark.parametrize("name", sorted(LDG))
def test_ldg_reads_constant_operands_only(name):
    for arg in re.findall(r"__ldg\((?:reinterpret_cast<[^>]*>\()?(\w+)", _text(name)):
        assert arg in LDG[name], (name, arg)
