"""The C-ABI library loads and exports every symbol the header declares (no compute, no GPU)."""
import ctypes
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared():
    text = open(os.path.join(ROOT, "include", "mpe.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(mpe_[a-z_0-9]+)\s*\(", text)))


def test_library_builds_and_exports_every_declared_symbol():
    from paper_2010_11305_b200 import build
    lib = ctypes.CDLL(build.build())
    names = _declared()
    assert {"mpe_create", "mpe_forward", "mpe_backward", "mpe_flush", "mpe_destroy", "mpe_step_host"} <= set(names)
    for n in names:
        assert hasattr(lib, n), f"{n} is declared in include/mpe.h but not exported"


def test_binding_covers_the_header():
    from paper_2010_11305_b200 import binding
    assert sorted(binding.EXPORTS) == _declared()


def test_product_path_has_no_oracle_dependency():
    pkg = os.path.join(ROOT, "paper_2010_11305_b200")
    for dirpath, _, files in os.walk(pkg):
        for f in files:
            if f.endswith((".py", ".cu", ".cuh", ".h")):
                src = open(os.path.join(dirpath, f)).read()
                assert not re.search(r"^\s*(from|import)\s+oracle|mpe_oracle|orc_[a-z]+\(", src, flags=re.M), f"{f} reaches into oracle/"


def test_create_fails_loudly_without_a_gpu():
    import torch
    from paper_2010_11305_b200 import binding
    if torch.cuda.is_available():
        return
    try:
        binding.Mpe([100], 16, 8, 0.1, 8, binding.LRU)
    except binding.MpeError as e:
        assert e.code == binding.ERR_CUDA
    else:
        raise AssertionError("mpe_create must not succeed without a CUDA device")


def test_error_codes_of_header_and_binding_agree():
    from paper_2010_11305_b200 import binding
    text = open(os.path.join(ROOT, "include", "mpe.h")).read()
    codes = dict(re.findall(r"\b(MPE_(?:OK|ERR_[A-Z_]+))\s*=\s*(-?\d+)", text))
    assert len(codes) >= 10
    for name, value in codes.items():
        short = name[len("MPE_"):]
        assert getattr(binding, short) == int(value), name


def test_bench_evidence_points_at_committed_summaries():
    """Every kernel record of the benchmark names the ncu summary its `bound` comes from: the file must be there, and it
    must be a text summary, nothing that runs."""
    import sys
    sys.path.insert(0, ROOT)
    import bench
    assert {"update", "pool", "hot_partial", "sort_scatter", "priority", "policy"} == set(bench.KERNEL_EVIDENCE)
    for name, ev in bench.KERNEL_EVIDENCE.items():
        path = os.path.join(ROOT, ev["profile"])
        assert os.path.isfile(path) and path.endswith(".md"), f"{name}: {ev['profile']}"
        assert "--clock-control none" in open(path).read(), f"{name}: the summary does not give its command"


def test_device_memory_is_cleared_in_front_of_its_first_use():
    """cudaMemset goes to the default stream, which a non-blocking stream does not wait for: the sort of a batch prepared on such a
    stream once counted in a workspace whose clear was still queued behind the running forward.  A clear either names the stream
    that uses the memory next, or the function it stands in waits for the device before it returns."""
    src = open(os.path.join(ROOT, "paper_2010_11305_b200", "csrc", "mpe.cu")).read()
    clears = [m.start() for m in re.finditer(r"\bcudaMemset\(", src)]
    assert clears
    for at in clears:
        rest = src[at:src.index("\n}\n", at)]
        assert "cudaDeviceSynchronize()" in rest, f"not waited for: {src[at:src.index(chr(10), at)]}"
    bench = open(os.path.join(ROOT, "bench.py")).read()
    made, switched = bench.index("stream_gen.batch(s) for s in"), bench.index("torch.cuda.set_stream(")
    assert "torch.cuda.synchronize(" in bench[made:switched]           # the batches are made on the default stream


def _source(name):
    return open(os.path.join(ROOT, "paper_2010_11305_b200", "csrc", name)).read()


def test_kernels_set_up_beside_their_predecessor_load_through_the_coherent_path():
    """A kernel that begins with after_previous_kernel() is resident while the kernel before it still writes; ld.global.nc and __ldg
    are for memory nobody writes meanwhile.  The one place left is k_update, which is launched when all before it has finished."""
    text = {f: _source(f) for f in ("mpe_device.cuh", "mpe_sort.cuh", "mpe_kernels.cuh", "mpe_table.cuh")}
    code = "".join(re.sub(r"//[^\n]*", "", t) for t in text.values())
    assert "ld.global.nc" not in code and code.count("__ldg(") == 1
    kernels = re.sub(r"//[^\n]*", "", text["mpe_kernels.cuh"])
    at = kernels.index("__ldg(")
    assert "k_update(State s" in kernels[kernels.rindex("__global__", 0, at):at]
    launched = set(re.findall(r'LAUNCH_NEXT\(h, "[a-z]+", (\w+)', _source("mpe.cu")))
    assert launched == {"kern", "k_priority"}                          # k_pool, k_update_small, k_priority (and k_table, by launch_table)


def test_waits_of_the_step_stream_are_known_to_its_launches():
    """A kernel behind an event the library makes the step's stream wait for is launched plainly: such waits go through one place."""
    src = _source("mpe.cu")
    assert src.count("cudaStreamWaitEvent(h->stream") == 1 and src.count("cudaStreamWaitEvent(st,") == 0
    assert src.count("ls.behind_kernel ?") == 2
