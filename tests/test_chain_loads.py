"""Kernels launched while their predecessor drains read, after the wait, memory
that the predecessor writes.  __ldg and const __restrict__ parameters promise that
nobody writes it during the kernel, so the compiler may load ahead of the wait: the
sources of such kernels, and of the stage bodies that they run, use neither."""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_1207_3392_gb300" / "csrc"


def _code(path):
    return re.sub(r"//[^\n]*", "", path.read_text())


def _chained_kernels():
    for path in sorted(CSRC.glob("*.cu*")):
        for text in re.split(r"__global__", _code(path))[1:]:
            if "{" not in text:  # a declaration
                continue
            head, body = text.split("{", 1)
            end = body.find("\n}")
            if "chain_wait()" in body[:end]:
                name = re.findall(r"(\w+)\s*\(", head.replace("__launch_bounds__(", "<"))[-1]
                yield f"{path.name}:{name}", head + body[:end]


KERNELS = dict(_chained_kernels())


def test_the_chained_kernels_are_found():
    names = " ".join(KERNELS)
    for k in ("hydro_strip_kernel", "hydro_strip_xy_kernel", "hydro_march_z_kernel",
              "finalize_kernel", "shock_flags_kernel", "init_from_primitive_kernel", "fmr_prolong_kernel",
              "fmr_child_faces_kernel", "mlp_reduce_adam_kernel"):
        assert k in names


@pytest.mark.parametrize("kernel", sorted(KERNELS))
def test_chained_kernels_promise_no_constant_memory(kernel):
    assert "__restrict__" not in KERNELS[kernel] and "__ldg" not in KERNELS[kernel]


def test_only_the_1d_tiles_join_the_chain():
    """The others read through __ldg."""
    code = _code(CSRC / "stage_kernel.cuh")
    assert "if constexpr (NDIM == 1) chain_wait();" in code and code.count("chain_wait") == 1
    assert "if constexpr (MARCH) return __ldg(p);" in code and code.count("__ldg") == 1
    assert "out->chain = NDIM == 1;" in _code(CSRC / "instantiate.cuh")


@pytest.mark.parametrize("name", ["stage_strip.cuh", "shock_flags.cuh", "fmr.cu", "aux_kernels.h"])
def test_bodies_of_chained_kernels_use_plain_loads(name):
    code = _code(CSRC / name)
    assert "__restrict__" not in code and "__ldg" not in code
