"""What the dependent launches (launch.cuh) rely on, read from the sources: which pointers of a kernel
that may start before its predecessor has ended are read-only for its whole life."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2104_04582_gb300", "csrc")

# const __restrict__ parameters of kernels launched by launch_pdl: data that no kernel before them on the
# stream can still be writing (the caller's arrays, complete before the plain launch just ahead; jobs
# uploaded and waited for when their batch was planned)
CONSTANT_INPUTS = {
    "k_build": {"jobs"},
    "k_direct_ring": {"pphi", "pr", "are", "aim"},
    "k_mode_select": {"amp_re", "amp_im"},
    "k_rb_pack_a": {"are", "aim"},
    "k_rb64_pack_a": {"are", "aim"},
}
# kernels that a launch_pdl reaches through a variable
BY_VARIABLE = {"kern": ["k_build", "k_build_one"], "kTc64Kernels[ks - 1]": ["k_sum_tc64"],
               "kTcKernels[ks - 1]": ["k_sum_tc"], "fp64 ? k_ylm<true> : k_ylm<false>": ["k_ylm"]}


def _source(name):
    with open(os.path.join(CSRC, name)) as fh:
        text = fh.read()
    return re.sub(r"//[^\n]*", "", text)


SOURCES = {f: _source(f) for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))}


def _dependent_kernels():
    names = set()
    for f, text in SOURCES.items():
        if f == "launch.cuh":
            continue
        for m in re.finditer(r"launch_pdl\(([^,]+),", text):
            names.update(BY_VARIABLE.get(m.group(1).strip(), [m.group(1).strip()]))
    return sorted(names)


@pytest.mark.parametrize("name", _dependent_kernels())
def test_no_read_only_path_to_what_a_predecessor_writes(name):
    found = 0
    for text in SOURCES.values():
        for m in re.finditer(r"__global__[^;{]*?\b" + name + r"\(([^{;]*?)\)\s*\{", text):
            found += 1
            const = set(re.findall(r"const \w+ ?\*\s*__restrict__ (\w+)", m.group(1)))
            assert const <= CONSTANT_INPUTS.get(name, set())
    assert found == 1


@pytest.mark.parametrize("name", ["tcsum.cu", "tcsum64.cu", "tctile.cuh", "fold_tc.cuh"])
def test_waveform_kernels_have_no_read_only_loads(name):
    # plans, records, tables, harmonics and spline data are all written by the kernel just before
    assert "__ldg(" not in SOURCES[name]
    for m in re.finditer(r"const [^;,()]*?\*\s*__restrict__ (\w+)", SOURCES[name]):
        assert m.group(1) == "kc"  # the block's own shared memory


def _launches(text):
    """The launches of a source in their order: 'plain', the dependent kernel's name, or 'checked'."""
    out = []
    for m in re.finditer(r"<<<|launch_pdl\(([^,]+),|(launch_rb64)\(|cudaGetLastError\(\)", text):
        out.append("plain" if m.group(0) == "<<<" else "checked" if m.group(0).startswith("cudaGet")
                   else (m.group(1) or m.group(2)).strip())
    return out


@pytest.mark.parametrize("name", [f for f in SOURCES if f.endswith(".cu")])
def test_plain_launch_is_checked_before_a_dependent_one(name):
    seq = _launches(SOURCES[name])
    for before, after in zip(seq, seq[1:]):
        assert not (before == "plain" and after not in ("plain", "checked"))


@pytest.mark.parametrize("name,kernel", [("rb.cu", "k_rb_pack_a"), ("rb.cu", "launch_rb64"), ("direct.cu", "k_direct_ring"),
                                         ("select.cu", "k_mode_select")])
def test_kernels_that_start_before_their_wait_follow_a_plain_launch(name, kernel):
    """They touch memory before their wait, which only a plain launch just ahead makes safe."""
    seq = [s for s in _launches(SOURCES[name]) if s != "checked"]
    assert seq[seq.index(kernel) - 1] == "plain"
