"""The stop flag of a Krylov loop. A kernel whose CTA 0 records the stop code may not read it from the same
place: the warps of a CTA that starts late could then read different values and part at a barrier. Read from
the sources: no function that several CTAs run both writes and reads one flag."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_1807_00086_gb300" / "csrc"
FLAG = r"(?:\*\s*o\.sc\.done|\*\s*sc\.done|\bo\.sc->done|(?<!\.)\bsc->done|\bo\.s[ct]->halt\[[^\]]*\]|\bsc->halt\[[^\]]*\])"


def _functions(text):
    """(name, body) of every function with a __global__ or __device__ qualifier"""
    text = re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))
    text = re.sub(r"__launch_bounds__\((?:[^()]|\([^()]*\))*\)", "", text)
    for m in re.finditer(r"__(?:global|device)__\b[^;{}]*?\b(\w+)\s*\([^;{}]*\)\s*(?:const\s*)?\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), text[m.end():i]


def _reads_and_writes(body):
    reads, writes = set(), set()
    for m in re.finditer(FLAG, body):
        name = re.sub(r"\s", "", m.group(0))
        (writes if re.match(r"\s*=(?!=)", body[m.end():]) else reads).add(name)
    return reads, writes


def test_no_grid_reads_the_stop_flag_that_it_writes():
    recorders = {}
    for path in sorted(CSRC.glob("*.cuh")):
        for name, body in _functions(path.read_text()):
            reads, writes = _reads_and_writes(body)
            if writes and "blockIdx" in body:
                recorders[name] = reads & writes
    assert {"cg_direction_kernel", "cg32_direction_kernel", "apply_two64_kernel", "cg2_begin_a",
            "cg2m_begin_a"} <= set(recorders)
    assert not {n: r for n, r in recorders.items() if r}


def test_the_scan_sees_a_flag_that_is_read_and_written():
    body = "if (o.sc->done) return; if (blockIdx.x == 0) o.sc->done = 1;"
    reads, writes = _reads_and_writes(body)
    assert reads & writes == {"o.sc->done"}
