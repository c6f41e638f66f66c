"""bench.py's bytes per node of a step, from the number of populations a node holds."""
import importlib.util
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_bytes_per_node():
    spec = importlib.util.spec_from_file_location("bench_bytes", os.path.join(ROOT, "bench.py"))
    bench = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(bench)
    assert bench.BYTES_PER_NODE == {"fp32": 2 * 27 * 4, "fp16": 2 * 27 * 2, "bf16": 2 * 27 * 2}
    assert bench.MHD_BYTES_PER_NODE == 2 * (27 + 3 * 7) * 4  # D3Q27 and, for three components, D3Q7
    assert bench.CG_BYTES_PER_NODE == 2 * (2 * 27) * 4 + 2 * 2 * 4  # two colours; (phi, rho) written and read
