"""A rebuild is due whenever a file that the library is compiled from has changed."""
import os


def test_every_source_file_is_a_dependency():
    from paper_1710_06316_gb300 import _build
    files = [os.path.join(_build.CSRC, f) for f in os.listdir(_build.CSRC) if f.endswith((".cu", ".cuh", ".h"))]
    files += [os.path.join(_build.INCLUDE, "afmpb.h")]
    assert set(files) <= set(_build.deps())
