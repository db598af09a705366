"""Rules that the kernels' sources keep, read from the sources."""
import glob
import os
import re

import paper_2604_11288_b200 as ta

CSRC = os.path.join(os.path.dirname(ta.__file__), "csrc")

# Kernels whose const __restrict__ inputs were written before another kernel of the same call, which lets its dependents start
# only when everything before it is complete.
BEHIND_OWN_KERNEL = {"ta_mask_kernel", "ta_ustatic_kernel", "ta_forced_kernel", "ta_select_kernel"}


def _kernels():
    """(name, parameters, body) of every kernel."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(([^)]*)\)\s*\{", src):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[end], 0)
                end += 1
            yield m.group(1), m.group(2), src[m.end():end]


def test_kernels_launched_early_read_no_callers_data_as_invariant():
    # a load through a const __restrict__ pointer may be moved above the wait for the kernel before this one
    seen = set()
    for name, params, body in _kernels():
        if "ta_wait_for_prior_grid()" not in body:
            continue
        seen.add(name)
        invariant = [p.strip() for p in params.split(",") if "__restrict__" in p and re.search(r"\bconst\b[^*]*\*", p)]
        assert not invariant or name in BEHIND_OWN_KERNEL, (name, invariant)
    first = {"ta_stream_step_kernel", "ta_embed_conf_kernel", "ta_compact_kernel", "ta_score_kernel", "ta_front_kernel"}
    assert first | BEHIND_OWN_KERNEL <= seen


def test_every_wait_takes_the_contexts_limit():
    # one place knows the default, no other file a limit of its own, and whoever has a context hands its limit on
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        if os.path.basename(path) != "ta_internal.cuh":
            assert not re.search(r"WaitLimitNs\b|\b2000000000", src), path
        if os.path.basename(path) == "ta_api.cu":
            made = re.findall(r"ta_select_args (\w+) = \{\};", src)
            assert made and all(f"{m}.wait_limit_ns = ctx->wait_limit_ns;" in src for m in made), made


def test_the_build_watches_every_header_that_a_source_includes():
    from paper_2604_11288_b200 import build
    watched = {os.path.basename(h) for h in build.headers()}
    for path in build.sources() + build.headers():
        for name in re.findall(r'#include "([^"]+)"', open(path).read()):
            assert os.path.basename(name) in watched, (path, name)
