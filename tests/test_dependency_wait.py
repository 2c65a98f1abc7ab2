"""Programmatic dependent launch, read from the sources: a kernel may start while the
kernels before it still run, so it touches what they write only after its wait
(pdl_enter), and takes the pointers it reads through past the compiler with after_wait
(loads through a ``const __restrict__`` argument may be moved above the wait)."""

import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2608_13578_gb300", "csrc")
# weights and the decay: inputs of the call that no kernel of this library writes
INPUTS = {"w_p", "W", "Wm", "decay"}
LOADS = r"\b(cp_async16|copy_rows16|ld_raw|load[48]\w*|ld_weight16|dec_cp16|__ldc?g)\s*\("


def _functions():
    """(file, name, parameter list, body) of every function whose body has pdl_enter()."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"\b(\w+)\s*\(((?:[^()]|\([^()]*\))*)\)\s*\{", src):
            if m.group(1) in ("if", "for", "while", "switch", "__launch_bounds__", "pdl_enter"):
                continue
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
            body = src[m.end():i - 1]
            if re.search(r"(?<!void )\bpdl_enter\(\);", body) and "__" in src[max(0, m.start() - 200):m.start()]:
                yield os.path.basename(path), m.group(1), m.group(2), body


FUNCTIONS = [f for f in _functions()]


def _base(expr, body):
    """The parameter a local pointer is formed from (``const T* dYb = dY + ...``)."""
    while True:
        m = re.search(r"\*\s*(?:const\s+)?%s = (\w+)\s*\+" % re.escape(expr), body)
        if not m:
            return expr
        expr = m.group(1)


def test_the_kernels_are_found():
    names = {f[1] for f in FUNCTIONS}
    assert {"gate_bwd_item", "summary_bwd_reg_kernel", "summary_bwd_kernel", "inject_kernel",
            "memory_proj_fwd_kernel", "gemm_simt_kernel", "decode_attn_kernel",
            "attn_bwd_dq_fl_kernel", "gemm_f32_kernel"} <= names


@pytest.mark.parametrize("file,name,params,body", FUNCTIONS, ids=lambda v: v if re.fullmatch(r"\w+", str(v)) else "")
def test_nothing_of_earlier_kernels_before_the_wait(file, name, params, body):
    before = body[:body.index("pdl_enter();")]
    pointers = set(re.findall(r"\*\s*(?:__restrict__\s+)?(\w+)", params))
    for stmt in re.split(r"[;{}]", before):
        reads = re.search(LOADS, stmt)
        for ident in re.findall(r"\b[A-Za-z_]\w*\b", stmt):
            p = _base(ident, body)
            if p not in pointers or p in INPUTS:
                continue
            indexed = re.search(r"\b%s\s*\[" % re.escape(ident), stmt)
            assert not reads and not indexed, (file, name, stmt.strip())


@pytest.mark.parametrize("file,name,params,body", FUNCTIONS, ids=lambda v: v if re.fullmatch(r"\w+", str(v)) else "")
def test_read_pointers_pass_after_wait(file, name, params, body):
    after = body[body.index("pdl_enter();"):]
    taken = {_base(p, body) for p in re.findall(r"after_wait\((\w+)\)", after)}
    for p in re.findall(r"const\s+[\w:]+\s*\*\s*__restrict__\s+(\w+)", params):
        # (a pointer that only goes on to a device function is that one's to take)
        assert p in taken or p in INPUTS or not re.search(r"\b%s\b" % p, body) or \
            re.search(r"_item<[^;]*\b%s\b" % p, body) and "gate_bwd" in name, (file, name, p)
