"""Read-only loads in kernels that are launched while their predecessor still
runs (launch_pdl): `ld.global.nc` (__ldg, or a const __restrict__ parameter)
asks for data that is constant for the whole life of the reading kernel, and
the predecessor may write until the reader's pdl_begin.  So in the source
files of those kernels it may only read what no predecessor writes: the scene
and the weights (written when they are loaded), and the march's records and
counts in the bucketing, which end two launches earlier (the scan between
them is launched after the march and starts with pdl_begin)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2208_02705_gb300", "csrc")

READ_ONLY = {
    "bucket.cu": {"recs", "cnt"},
    "march.cu": {"g.brick_dist", "g.cells", "g.labels"},
    "mlp_simt.cu": {"wf"},
    "mlp_tc.cu": {"aff"},
}


def _sources():
    return {os.path.basename(p): open(p).read() for p in sorted(glob.glob(os.path.join(CSRC, "*.cu")))}


def _argument(src, at):
    """The text between the parenthesis at src[at] and its partner."""
    depth = 0
    for i in range(at, len(src)):
        depth += {"(": 1, ")": -1}.get(src[i], 0)
        if depth == 0:
            return src[at + 1:i]
    raise AssertionError("unbalanced parentheses")


def _pointer(arg):
    """The pointer that an address expression starts from."""
    arg = re.sub(r"reinterpret_cast<[^>]*>", "", arg)
    return re.match(r"[(&\s]*([A-Za-z_][\w.]*)", arg).group(1)


def test_read_only_loads_name_constant_data():
    seen = set()
    for name, src in _sources().items():
        if "launch_pdl(" not in src:
            continue
        for m in re.finditer(r"__ldg\(", src):
            p = _pointer(_argument(src, m.end() - 1))
            assert p in READ_ONLY.get(name, ()), f"{name}: __ldg of {p}, which a running predecessor may write"
            seen.add((name, p))
        assert "ld.global.nc" not in src, name
    assert seen == {(f, p) for f, ps in READ_ONLY.items() for p in ps}


def test_kernels_launched_early_have_no_restrict_parameters():
    """(the compiler may turn loads through const __restrict__ parameters into
    read-only ones)"""
    checked = set()
    for name, src in _sources().items():
        for kernel in re.findall(r"launch_pdl\(\s*(?:[^,?]*\?\s*)?(k_\w+)", src):
            for m in re.finditer(r"__global__[^;{]*?\b%s\(" % kernel, src):
                assert "__restrict__" not in _argument(src, m.end() - 1), (name, kernel)
                checked.add(kernel)
    assert {"k_scan", "k_scatter_blk", "k_march", "k_composite_round", "k_mlp_simt", "k_mlp_tc"} <= checked
