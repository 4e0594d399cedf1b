"""A kernel's shared-memory limit (cudaFuncSetAttribute) belongs to one device's
copy of the kernel: it is set on every path to a launch, never behind a flag
that the process keeps, or a frame on a second device of the process is
refused.  One device cannot show that at run time, so the sources are read."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2201_05497_gb300" / "csrc"
DEFAULT_LIMIT = 48 * 1024


def body(text, start):
    """text from `start` to the end of the brace block that opens after it."""
    depth = 0
    for i in range(text.index("{", start), len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[start:i + 1]
    raise AssertionError("unbalanced braces")


def test_no_attribute_is_kept_by_the_process():
    """No function that a call_once or a static flag guards raises the limit
    above the default, directly or through a helper of its file."""
    found = 0
    for path in sorted(CSRC.glob("*.cu")):
        text = re.sub(r"//[^\n]*", "", path.read_text())
        found += text.count("cudaFuncSetAttribute(")
        guarded = [body(text, m.start()) for m in re.finditer(r"std::call_once\(", text)]
        guarded += [body(text, m.start()) for m in re.finditer(r"\nvoid \w+\(\)\s*\{\s*static bool", text)]
        for g in guarded:
            # the persistent kernel's table is 16 KB: any device launches it without the attribute
            if "persist_epoch_kernel" in g:
                assert "(lmh::TOF_TAB_N + 1) * 4" in g and 4097 * 4 <= DEFAULT_LIMIT
                continue
            assert "cudaFuncSetAttribute" not in g, (path.name, g)
        # a guarded occupancy count may raise the limit on its way, if every launch does so too
        for name in re.findall(r"(\w+_kernel\w*)(?:<[^<>]*>)?<<<[^;]*TAB_SMEM", text):
            assert re.search(r"table_smem\(" + name, text) or name == "kernel", (path.name, name)
    assert found >= 8
