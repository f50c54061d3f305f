"""Forms of the copy engine that the kernels must not use: a load that one CTA
issues into several CTAs of its cluster is only for code that runs on one GPU
alone, and this library also runs as replicas, one per GPU (`bench.py --gpus`)."""
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_load_into_several_ctas():
    word = "multi" + "cast"
    found = []
    for d in ("paper_2404_13811_gb300", "include"):
        for base, dirs, files in os.walk(os.path.join(ROOT, d)):
            dirs[:] = [x for x in dirs if not x.startswith(("_build", "__pycache__"))]
            for fn in files:
                if fn.endswith((".cu", ".cuh", ".h", ".py")):
                    with open(os.path.join(base, fn)) as f:
                        found += [f"{fn}:{i}" for i, line in enumerate(f, 1) if word in line.lower()]
    assert not found, found
