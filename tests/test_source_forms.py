"""Forms that the kernels must not use.  Of the copy engine: a load that one CTA
issues into several CTAs of its cluster is only for code that runs on one GPU
alone, and this library also runs as replicas, one per GPU (`bench.py --gpus`).
Of the conversions to FP32: truncation in the 3D kernels."""
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


def test_3d_kernels_round_to_nearest():
    """The couplings that stay in a box's factor and the residuals its sweeps take
    are rounded, as an FP32 cast would (d2f_bits truncates); pivots are divided by
    the correctly rounded reciprocal."""
    csrc = os.path.join(ROOT, "paper_2404_13811_gb300", "csrc")
    with open(os.path.join(csrc, "local3d.cu")) as f:
        assert "d2f_bits(" not in f.read()
    with open(os.path.join(csrc, "box2d.cuh")) as f:
        body = f.read().split("float rcp_piv(float v)")[1].split("}")[0]
    assert "__frcp_rn" in body, body
