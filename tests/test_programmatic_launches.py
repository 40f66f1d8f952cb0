"""Kernels launched with programmatic dependence start while the kernel before them still runs, and only
griddepcontrol.wait makes what it wrote visible: every such kernel waits before it touches memory.  Read from the
sources: the launches go through one helper, the wait stands in one function, and the text of each kernel that the
helper launches has no memory access, return or barrier before that function's call."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1506_07656_gb300", "csrc")
SOURCES = {os.path.basename(p): re.sub(r"//[^\n]*", "", open(p).read()) for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*")))}


def test_one_helper_and_one_wait():
    launches = {f: len(re.findall(r"cudaLaunchKernelEx\b|ProgrammaticStreamSerialization\b", s)) for f, s in SOURCES.items()}
    waits = {f: len(re.findall(r"griddepcontrol|cudaGridDependencySynchronize|cudaTriggerProgrammatic", s))
             for f, s in SOURCES.items()}
    assert {f: n for f, n in launches.items() if n} == {"dm_internal.cuh": 2}
    assert {f: n for f, n in waits.items() if n} == {"dm_internal.cuh": 2}


def _kernels():
    """(file, kernel) of every launch through the helper; a local alias is resolved to the kernels it names."""
    found = set()
    for f, s in SOURCES.items():
        for m in re.finditer(r"\bdm_launch_pdl\(\s*(\w+)", s):
            name = m.group(1)
            if name == "void":                            # the helper's own definition
                continue
            alias = re.findall(r"\bauto %s = ([^;]*);" % name, s)
            for k in (re.findall(r"\bk_\w+", alias[-1]) if alias else [name]):
                found.add((f, k))
    return sorted(found)


def _body(source, kernel):
    """Pointer parameters of a __global__ function and the text of its body."""
    m = re.search(r"__global__[^;{]*?\b%s\(([^{]*)\)\s*\{" % kernel, source)
    assert m, kernel
    params, body = m.group(1), source[m.end():]
    body = body[:re.search(r"\n\}", body).start()]
    assert "dm_pdl_wait();" in body, f"{kernel} does not wait"
    return re.findall(r"\*\s*(?:__restrict__\s*)?(\w+)", params), body


def test_every_kernel_waits_first():
    kernels = _kernels()
    assert {"k_df_sor_tb", "k_level_rows", "k_level_top", "k_bt_expand", "k_descriptors"} <= {k for _, k in kernels}
    for f, k in kernels:
        pointers, body = _body(SOURCES[f], k)
        if k == "k_df_sor_tb":                            # stages ahead of the wait: below
            continue
        head = body[:body.index("dm_pdl_wait();")]
        for p in pointers:
            assert not re.search(r"\b%s\b" % p, head), f"{k} uses {p} before it waits"
        # members of argument structs that point to memory (lower-case scalars of a geometry are values)
        assert not re.search(r"\ba\.(hdr|valid|pooled|amax|best\w+|keys|slots|v)\b", head), k
        assert not re.search(r"__ldg|__ldcg|\breturn\b|\bif\b|__syncthreads|\batomic", head), k


def test_reads_ahead_of_the_wait_are_acquired():
    """The blocked SOR launches read u, v, ps and A before their wait, after an acquire of the count that the
    kernel writing them publishes by a release (else they wait first); the increments, which the launch
    before writes, only after the wait."""
    source = SOURCES["k_deepflow.cu"]
    _, body = _body(source, "k_df_sor_tb")
    first = body.index("const bool early = count != 0u && df_acquired(published, count);\n    if (!early) dm_pdl_wait();")
    last = body.index("if (early) dm_pdl_wait();")
    assert body.count("dm_pdl_wait();") == 2 and first < last
    reads = {m: [x.start() for x in re.finditer(r"\bL\.%s\b" % m, body)] for m in ("u", "v", "ps", "A", "du", "dv")}
    assert all(reads[m] and min(reads[m]) > first for m in ("u", "v", "ps", "A"))
    assert all(reads[m] and min(reads[m]) > last for m in ("du", "dv"))
    assert "out_du" not in body[:last] and "out_dv" not in body[:last]
    assert "ld.acquire.gpu" in source and re.search(r"__syncthreads\(\);\s*if \(threadIdx\.x == 0\) asm volatile\(\"red\.release\.gpu", source)
