"""Kernels of a launch chain (csrc/chain.cuh) are resident while the kernel before
them writes.  PTX defines non-coherent loads (__ldg, and loads from parameters that
are both const and __restrict__) only for memory that is not written during the
kernel's whole life, so such kernels may use them for links, and for the shadow
vector r_hat (aux), which only kernels outside the chain write.  Read off the
sources: the kernels that call chain_enter(), and every device helper."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0710_1988_gb300", "csrc")
LINKS = {"links", "L", "aux", "rhat"}
# helpers that load links or r_hat, or serve only kernels outside the chain (the FP64 stencils, the encoder of a whole vector)
LINK_HELPERS = {"ld_fixed32", "ld_fixed16", "ld_link32", "ld_link16", "ld_link_eo", "fx_terms", "fx_pair_f64", "su3_mul", "su3_adj_mul_acc",
                "su3_mul_eo"}
UNCHAINED_HELPERS = {"load_spinor", "hop_eo"}


def _functions(text):
    """(qualifier, name, parameters, body) of every function with a body."""
    for m in re.finditer(r"(__global__|__device__)[^;{]*?\b(\w+)\(([^{};]*?)\)\s*\{", text):
        name = [w for w in re.findall(r"(\w+)\(", text[m.start():m.end()]) if w != "__launch_bounds__"][0]
        i, depth = m.end(), 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        head = text[m.start():m.end()]
        yield m.group(1), name, head[head.index(name):], text[m.end():i]


def _all():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for fn in _functions(text):
            yield (os.path.basename(path),) + fn


def test_chained_kernels_read_vectors_by_ordinary_loads():
    chained = [fn for fn in _all() if fn[1] == "__global__" and "chain_enter()" in fn[4]]
    assert len(chained) >= 15
    for path, _, name, params, body in chained:
        loose = set(re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", params)) - LINKS
        assert not loose, (path, name, loose)
        for arg in re.findall(r"__ldg\(\s*(?:reinterpret_cast<[^>]*>\()?(\w+)", body):
            assert arg in LINKS | {"l", "ab"}, (path, name, arg)    # pointers into the links, aux


def test_helpers_of_chained_kernels_read_vectors_by_ordinary_loads():
    kernels = {n for _, q, n, _, b in _all() if q == "__global__" and "chain_enter()" in b}
    bodies = {n: b for _, _, n, _, b in _all()}
    reach, todo = set(), list(kernels)
    while todo:                                  # functions called from a chained kernel
        for callee in re.findall(r"\b(\w+)\s*(?:<[^;(){}]*>)?\(", bodies[todo.pop()]):
            if callee in bodies and callee not in reach:
                reach.add(callee)
                todo.append(callee)
    assert "ld_spinor32" in reach and "ld_h" in reach
    assert not reach & UNCHAINED_HELPERS
    for name in reach - kernels:
        if "__ldg(" in bodies[name]:
            assert name in LINK_HELPERS, name
