"""The rule of the kernels that are launched with a programmatic dependency (internal.h): such a kernel is resident while the one before
it in the stream may still write its inputs.  `const ... __restrict__` on a kernel parameter promises memory that nobody writes for the
kernel's whole life, which lets the compiler load it before the wait and past the coherent caches; it is therefore kept to the tables a
context builds once."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_21131_b200", "csrc")
TABLES = {"lt", "keytab"}  # constants of the limbs, addresses of the loaded keys


def chained_kernels():
    """(file, name, parameter list) of every kernel whose body waits for its predecessor"""
    out = []
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith(".cu"):
            continue
        text = open(os.path.join(CSRC, f)).read()
        for m in re.finditer(r"__global__ void (?:__launch_bounds__\((?:[^()]|\([^()]*\))*\) )?(\w+)\(([^{]*?)\) \{\n(.*?)\n\}\n", text, re.S):
            if "chain_wait();" in m.group(3):
                out.append((f, m.group(1), m.group(2)))
    return out


def test_inputs_of_chained_kernels_are_not_promised_to_be_constant():
    kernels = chained_kernels()
    assert len(kernels) >= 18 and {"k_linear", "k_mac_bulk", "k_ks_inner_stream", "k_ks_apply"} <= {k for _, k, _ in kernels}
    bad = [(f, k, name) for f, k, params in kernels for name in re.findall(r"const [\w ]+\*(?: const\*)? __restrict__ (\w+)", params)
           if name not in TABLES]
    assert not bad, bad
