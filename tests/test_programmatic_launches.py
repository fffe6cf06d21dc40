"""Kernels that start before the launch ahead of them has ended (those that
call grid_dep_wait), read as source.  What earlier launches write is read with
ordinary loads: a read-only load (__ldg, or a const __restrict__ kernel
argument, which the compiler may turn into one) is for memory that nothing
writes while the kernel runs, which here begins before its wait, so it is left
to the tables."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1011_3582_gb300", "csrc")
# written by fftlb_create alone
TABLES = {"tw_g", "Wh_g", "Wp_g", "kxt", "A.kx", "A.ky", "src"}   # src: load_tab4 (tables to shared memory)


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def closing(text, i, pair):
    """Index after the bracket that closes the one before index i."""
    depth = 1
    while depth:
        depth += {pair[0]: 1, pair[1]: -1}.get(text[i], 0)
        i += 1
    return i


def kernels():
    """(name, parameters, body) of every __global__ function."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = source(os.path.basename(path))
        for m in re.finditer(r"__global__\s+void\s+(__launch_bounds__\s*\()?", text):
            at = closing(text, m.end(), "()") if m.group(1) else m.end()
            name = re.compile(r"\s*(\w+)\(").match(text, at)
            args = closing(text, name.end(), "()")
            body = text.index("{", args) + 1
            out.append((name.group(1), text[name.end():args - 1], text[body:closing(text, body, "{}")]))
    return out


def waiting():
    ks = [k for k in kernels() if "grid_dep_wait" in k[2]]
    names = {k[0] for k in ks}
    assert {"k1_row", "k3_row", "k5_row", "k1_wr", "k3_wr", "k5_wr", "kcol_reg", "kcol_line", "energy_row", "energy_col",
            "energy_line", "k_inv_sites", "k_reduce_partials"} <= names
    return ks


def test_read_only_loads_are_of_tables():
    for name, params, body in waiting():
        for arg in re.findall(r"const\s+[\w:<>]+\s*\*\s*__restrict__\s+(\w+)", params):
            assert arg in TABLES, (name, arg)
    for f in ("kernels_row.cuh", "kernels_wr.cuh", "kernels_col.cuh"):
        for arg in re.findall(r"__ldg\(([\w.]+)", source(f)):
            assert arg in TABLES or arg == "p" and f == "kernels_col.cuh", (f, arg)   # p: tab(), a table value


def test_copies_of_the_stage_follow_the_wait():
    """Only tables are copied to shared memory before grid_dep_wait."""
    for name, _, body in waiting():
        before = body[:body.index("grid_dep_wait")]
        for call in re.findall(r"\b(\w*(?:issue\w*|bulk_\w+|prefetch\w*|tma_\w+))(?:<[\w, ]+>)?\(", before):
            assert call in ("table_issue", "issue"), (name, call)   # issue: ColTab's
