"""Kernels that may be placed on the SMs while the kernels before them still
write the fields (those that call pdl_wait) read these fields through coherent
loads only. What a wrong load reads depends on what an SM's cache holds, so
this is checked in the sources and not by running it."""
import glob
import os
import re

import paper_1603_03971_gb300

CSRC = os.path.join(os.path.dirname(paper_1603_03971_gb300.__file__), "csrc")
# written before a call's first step, or by nobody, while such a kernel lives
STABLE = {"c", "rec", "taps", "r_row", "coarse"}
FIELDS = r"\b(u_cur|u_prev|mu_cur|mu_prev|snap|acc|slab|illum|band|field|prev|cur|u)\b"
READ_ONLY = re.compile(r"\b(__ldg|ld_keep|vld_keep\w*(?:<\w+>)?)\s*\(([^;]*)")


def _kernels():
    """(name, parameter list, body) of every kernel that calls pdl_wait()."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        with open(path) as f:
            src = re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)
        for m in re.finditer(r"__global__\s+void\b[^{;]*?\b(k_\w+)\s*\(", src):
            depth, i = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(src[i], 0)
                i += 1
            params, body = src[m.end():i - 1], src.index("{", i)
            depth, j = 1, body + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[j], 0)
                j += 1
            if "pdl_wait()" in src[body:j]:
                yield m.group(1), params, src[body:j]


def test_early_placed_kernels_read_fields_coherently():
    names = []
    for name, params, body in _kernels():
        names.append(name)
        for p in params.split(","):
            if "__restrict__" in p:
                assert p.split()[-1] in STABLE, (name, p.strip())
        for m in READ_ONLY.finditer(body):
            assert not re.search(FIELDS, m.group(2)), (name, m.group(0).strip())
    # the kernels of a time step are all among them
    for k in ("k_stencil_tma", "k_stencil_rows", "k_fwd_aux", "k_bwd_aux", "k_fwd_aux_off",
              "k_bwd_aux_off", "k_band_copy", "k_illum_add", "k_decimate", "k_upsample",
              "k_encode_march"):
        assert k in names, k


def test_weights_read_before_the_wait_follow_an_ordinary_launch():
    """k_encode_march reads its weights before the wait: the first kernel of
    the scale, which precedes it, is an ordinary launch on either path."""
    with open(os.path.join(CSRC, "ae.cu")) as f:
        src = f.read()
    assert re.search(r"k_sumsq<<<[^>]*>>>\(in", src)
    ready = src[src.index("if (sumsq_ready)"):]
    assert re.match(r"if \(sumsq_ready\) \{\s*k_scale<<<", ready)
