"""Kernels launched by launch_chained may be resident while the kernel before them still
writes the fields they read, so only data that no kernel of a chain writes, the links
and the clover blocks, may go through the read-only path (__ldg, ld.global.nc): its
loads need data that stay unchanged for as long as the kernel exists, and the compiler
may move them across the wait.  Checked on the sources of the chained kernels and the
headers they share."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_2212_06635_gb300" / "csrc"

def _code(path):
    src = re.sub(r"/\*.*?\*/", "", path.read_text(), flags=re.S)
    return re.sub(r"//[^\n]*", "", src)


def _functions(src):
    """(name, body) of every function and kernel, lambdas inside their function."""
    src = re.sub(r"__launch_bounds__\((?:[^()]|\((?:[^()]|\([^()]*\))*\))*\)", "", src)
    out, end = [], 0
    for m in re.finditer(r"\b(\w+)\s*\([^;{}]*\)\s*\{", src):
        if m.start() < end or m.group(1) in ("if", "for", "switch", "while"):
            continue
        depth, k = 1, m.end()
        while depth and k < len(src):
            depth += {"{": 1, "}": -1}.get(src[k], 0)
            k += 1
        end = k
        kernel = "__global__" in src[max(0, src.rfind("}", 0, m.start()), src.rfind(";", 0, m.start())):m.start()]
        out.append((m.group(1), src[m.end():k], kernel))
    return out


def _chained():
    """(file, function, body): the kernels handed to launch_chained and all functions
    that are not kernels, of the files that launch them and of the headers they share."""
    headers = [CSRC / "tm_internal.h", CSRC / "tm_kernels.h", CSRC / "dslash_common.cuh"]
    launches, found = set(), []
    for path in sorted(CSRC.glob("*.cu")) + headers:
        src = _code(path)
        names = set(re.findall(r"launch_chained\(\s*(\w+)\s*<", src))
        if not names and path.suffix == ".cu":
            continue
        launches |= names
        found += [(path.name, f, body) for f, body, kernel in _functions(src) if not kernel or f in names]
    assert launches >= {"dslash_kernel", "dslash_heavy_kernel", "dslash_pair_kernel", "dslash_split_kernel",
                        "dslash_dw_kernel", "dslash_staged_kernel", "k_cg_direction"}
    assert launches <= {f for _, f, _ in found}
    return found


def test_the_read_only_path_is_taken_in_one_function():
    inside = {f for _, f, body in _chained() if "__ldg(" in body}
    assert inside == {"load_vec"}


def test_only_links_and_clover_blocks_are_read_through_it():
    """Every call that names the read-only path, and load_link, which always takes it."""
    seen = set()
    read_only = re.compile(r"(load_readonly|load_link|load_herm_row|load_\w+<[^;()]*\btrue>)\s*(?:<[^;()]*?>)?\s*\(([^;]*);")
    for name, f, body in _chained():
        for m in read_only.finditer(body):
            args = m.group(2).strip()
            if m.group(1).startswith("load_vec") and f == "load_link":
                continue   # the path itself
            if m.group(1) == "load_herm_row":   # (destination, array, ...)
                args = args.split(",", 1)[1].strip()
            if f in ("load_readonly", "load_herm_row") and args.startswith("base"):
                continue
            assert re.match(r"pr\.(gauge\[|clov\b)", args), (name, f, m.group(0)[:80])
            seen.add(name)
    assert seen >= {"dslash.cu", "dslash_heavy.cu", "dslash_split.cu"}


def test_clover_reads_before_the_wait_are_read_only_data():
    """What the split kernel loads before it waits for the kernel before it."""
    src = _code(CSRC / "dslash_split.cu")
    kernel = src[src.index("dslash_split_kernel("):]
    early = kernel[:kernel.index("pdl_wait()")]
    assert "pr.clov" in early
    assert not re.search(r"pr\.(in|loc|out|r|p)\b", early)
