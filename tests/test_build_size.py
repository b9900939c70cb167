"""The libraries and objects that the build leaves in the tree stay small enough
to ship a checkout with them: the bounds-checked variant's device code is
compressed (build.py)."""
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LIMIT = 400 << 20  # the ordinary and the bounds-checked build together


def test_build_products_stay_below_the_limit():
    import paper_2506_07793_gb300  # noqa: F401  (refuses to import without its library)
    total = 0
    for sub in ("_build", "_build_check", "_lib"):
        for base, _, files in os.walk(os.path.join(ROOT, "paper_2506_07793_gb300", sub)):
            total += sum(os.path.getsize(os.path.join(base, f)) for f in files)
    assert 0 < total <= LIMIT, f"{total >> 20} MB of build products"
