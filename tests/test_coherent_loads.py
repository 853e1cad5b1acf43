"""__ldg reads through the non-coherent path, whose data must be read-only for the lifetime of the kernel.  Kernels of
the solver may begin while the one before them still writes (programmatic dependent launch) and the operator may run
in place, so __ldg is for tables, spectra and the potential only, in every kernel that is launched that way."""
import os
import re

CSRC = os.path.join("paper_1910_13844_gb300", "csrc")
# stage twiddles; the Green values and far-field kernels; the fused pass's column order; the potential
TABLES = {"a.tw", "a.tw2", "tw4", "twb4", "a.zwa", "a.zwb", "a.ytw", "a.ztw", "a.cols", "a.gocta", "col", "gc", "k", "f"}


def _kernels(text):
    """(name, body) of every function in a source file, split at column-0 'template' / '__global__' / '__device__'."""
    for part in re.split(r"\n(?=template|__global__|__device__|static|inline|struct)", text):
        m = re.search(r"\b(k_\w+|\w+_body|fx_store)\s*\(", part)
        yield (m.group(1) if m else ""), part


def test_ldg_reads_tables_only(repo_root):
    launched, seen = set(), 0
    sources = {}
    for name in sorted(os.listdir(os.path.join(repo_root, CSRC))):
        if name.endswith((".cu", ".cuh")):
            sources[name] = open(os.path.join(repo_root, CSRC, name)).read()
            launched |= set(re.findall(r"launch_pdl\([^;]*?\b(k_\w+)", sources[name]))
    assert {"k_fx", "k_ix", "k_update", "k_far_reduce", "k_yz"} <= launched
    for name, text in sources.items():
        whole = name in ("passes.cuh", "yz.cuh", "zpass.cuh")
        for kernel, body in _kernels(text):
            if not whole and kernel not in launched:
                continue
            for arg in re.findall(r"__ldg\(\s*([\w.]+)", body):
                seen += 1
                assert arg in TABLES, (name, kernel, arg)
    assert seen > 20
