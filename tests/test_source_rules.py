"""Rules that the kernels' sources keep (igg_internal.h states the reasons)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2211_15716_gb300", "csrc")
# tables that no launch writes; memory that the kernels only store to
TABLES = {"tiles", "copies", "nbr"}
STORED = {"T2", "lam_out", "gCi", "fix", "dev_err"}


def _kernels():
    """(file, kernel name, parameter list, body) of every kernel."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = open(path).read()
        for m in re.finditer(r"__global__ void(?:\s+__launch_bounds__\([^{;]*?\))?\s+(k_\w+)\(", src):
            i, depth = m.end(), 1
            while depth:
                depth += {"(": 1, ")": -1}.get(src[i], 0)
                i += 1
            params, j = src[m.end():i - 1], src.index("{", i)
            k, depth = j + 1, 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[k], 0)
                k += 1
            yield os.path.basename(path), m.group(1), params, src[j:k]


def test_kernels_are_found():
    names = {k[1] for k in _kernels()}
    assert {"k_stencil_tma", "k_stencil_rows", "k_fixup_f64", "k_adjoint_tma", "k_gp_tma",
            "k_acoustic_v", "k_acoustic_p", "k_halo_gather", "k_halo_jobs"} <= names


def test_no_restricted_reads_behind_the_dependency_wait():
    for file, name, params, body in _kernels():
        if "pdl_wait()" not in body:
            continue
        restricted = set(re.findall(r"__restrict__\s+(\w+)", params))
        assert restricted <= TABLES | STORED, (file, name, restricted - TABLES - STORED)
        for p in restricted & STORED:  # (reads through the pointer itself)
            assert not re.search(r"=\s*\*?%s\s*\[" % p, body), (file, name, p)
        assert "__ldg" not in body, (file, name)


def test_stores_of_the_stencils_are_bounds_checked():
    """Every function of the stencil that stores to T2 tests its index in the
    bounds-checked build."""
    seen = 0
    for file in ("tma.cu", "rows.cu"):
        src = open(os.path.join(CSRC, file)).read()
        for m in re.finditer(r"^(?:template <[^>]*>\n)?__(?:global|device)__[^;{]*?(\w+)\([^;{]*\{\n(.*?)^\}",
                             src, re.M | re.S):
            body = m.group(2)
            if re.search(r"(T2|d0|dst)(\[[^\]]*\])+ = |\*reinterpret_cast<uint4 \*>\(dst\) =", body):
                seen += 1
                assert "in_bounds(" in body, (file, m.group(1))
    assert seen >= 4  # k_stencil_tma, emu_fix_rows, k_fixup_f64, k_stencil_rows
