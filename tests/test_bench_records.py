"""The bench's captured figures are tied to the sources that they were captured with."""
import glob
import importlib.util
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2507_09165_gb300", "csrc")
# translation units that take no part in a single projection
APART = {"batched.cu", "batched_kernels.cu", "deflate.cu", "noalloc.cu", "server.cu"}


def test_tensor_pipe_sources_cover_the_single_projection():
    spec = importlib.util.spec_from_file_location("bench_mod", os.path.join(ROOT, "bench.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    files = {os.path.basename(p) for ext in ("*.cu", "*.cuh", "*.h") for p in glob.glob(os.path.join(CSRC, ext))}
    assert set(m.TENSOR_PIPE_SOURCES) == files - APART
