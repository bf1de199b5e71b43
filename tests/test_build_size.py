"""The built tree (objects and library, all kernel variants) stays small enough to be copied
around with the sources: 256 MB, where line tables alone once took 400."""
import glob
import os


def test_built_files_stay_below_256_mb():
    from paper_1804_08593_gb300 import build
    files = [build.build()] + glob.glob(os.path.join(build.BUILD, "*.o"))
    assert len(files) > 60
    size = sum(os.path.getsize(f) for f in files)
    assert size < 256 << 20, size
