"""bench.py names the kernel that each GEMM option launches."""

import os
import re

import bench

CSRC = os.path.join(os.path.dirname(os.path.abspath(bench.__file__)), "paper_1911_12954_gb300", "csrc")


def _text(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def test_kernel_names_follow_the_dispatch():
    host, tc = _text("hotrg.cu"), _text("gemm_tc.cu")
    # launch_gemm_group: variant number -> configuration
    body = tc[tc.index("cudaError_t launch_gemm_group("):]
    cfg = {int(v): (kind, c) for v, kind, c in
           re.findall(r"if \(variant == (\d)(?: && dv->pair_grid >= 2)?\)\s*return launch_(single|pair)<(\w+)>", body)}
    pair5 = re.search(r"if \(dv->pair_grid >= 2\) return launch_pair<(\w+)>", body).group(1)
    cfg[5] = ("pair", pair5)
    for precision, table in (("fp16x3", "kF16Variant"), ("tf32x3", "kTF32Variant")):
        variants = [int(x) for x in re.search(table + r"\[\d\] = \{([^}]*)\}", host).group(1).split(",")]
        for option, v in enumerate(variants):
            kind, c = cfg[v]
            kernel = {"pair": "gemm_pair_kernel", "single": "gemm_tf32x3_kernel"}[kind]
            assert bench.kernel_name(precision, option).startswith("%s<%s>" % (kernel, c)), (precision, option)
