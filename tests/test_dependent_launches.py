"""What the warm-start kernels' overlap rests on, read from their source (the
faults these rules keep out would hang or fault a GPU, so nothing here runs).

Every kernel of a network pass is a programmatic dependent of the one before:
it may be resident while that one runs, until its dependency_wait() returns."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_04446_gb300", "csrc")


def _kernels():
    """{name: (parameters, body)} of the __global__ functions of the network, comments removed."""
    out = {}
    for name in ("conv_umma.cuh", "warmstart.cu"):
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for m in re.finditer(r"__global__ void (?:__launch_bounds__\([^()]*\)\s*)?(\w+)\(", src):
            i, depth = m.end(), 1
            while depth:
                depth += {"(": 1, ")": -1}.get(src[i], 0)
                i += 1
            params = src[m.end():i - 1]
            i = j = src.index("{", i)
            depth = 0
            while True:
                depth += {"{": 1, "}": -1}.get(src[j], 0)
                j += 1
                if depth == 0:
                    break
            out[m.group(1)] = (params, src[i:j])
    return out


KERNELS = _kernels()


def test_the_kernels_were_found():
    assert {"conv_gemm_kernel", "finish_split_kernel", "conv_first_kernel", "conv_first_wgrad_kernel",
            "mask_split_kernel", "sum_slices_kernel", "pack_wmats_kernel", "mse_kernel", "adam_kernel"} <= set(KERNELS)


@pytest.mark.parametrize("name", sorted(KERNELS))
def test_every_kernel_triggers_and_waits_once(name):
    body = KERNELS[name][1]
    assert body.count("dependency_trigger()") == 1 and body.count("dependency_wait()") == 1


@pytest.mark.parametrize("name", sorted(k for k in KERNELS if "tcgen05.alloc" in KERNELS[k][1]))
def test_dependents_start_after_the_tensor_memory_is_allocated(name):
    body = KERNELS[name][1]
    alloc, trigger = body.index("tcgen05.alloc"), body.index("dependency_trigger()")
    assert alloc < trigger and "__syncthreads()" in body[alloc:trigger]


def test_both_issuing_roles_drain_whatever_role_gave_up():
    """The last copies (full barriers) and the last MMAs (empty barrier) are waited for
    without a look at whether this role's own waits succeeded."""
    body = KERNELS["conv_gemm_kernel"][1]
    loops = body.index("if (warp == 0)")
    for bar in ("full", "empty"):
        waits = [m.start() for m in re.finditer(r"mbar_drain\(&%s\[" % bar, body)]
        assert len(waits) == 1 and waits[0] > loops
        statement = body[max(body.rfind(c, 0, waits[0]) for c in "{}"):waits[0]]
        assert "ok" not in statement


@pytest.mark.parametrize("name", sorted(KERNELS))
def test_no_load_takes_the_non_coherent_path(name):
    """A buffer that an earlier kernel of the pass may still write is not read-only for the
    reading kernel's lifetime: no __ldg, no const __restrict__ parameter, no plain
    dereference that a compiler could turn into either (umma::ld is volatile)."""
    params, body = KERNELS[name]
    assert "__ldg" not in body and "__restrict__" not in params
    pointers = re.findall(r"const (?:float|__nv_bfloat16)\s*\*\s*(\w+)", params)
    for p in pointers:
        assert not re.search(r"\b%s\[" % p, body), p


def test_gemm_splits_follow_the_device():
    """How many K slices a GEMM gets depends on the SMs that its persistent CTAs run on,
    which are read from the device: no SM count in the rule."""
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "warmstart.cu")).read())
    assert re.findall(r"[^\n]*\b152\b[^\n]*", src) == ["constexpr int kBiasSlices = 152;     "]
