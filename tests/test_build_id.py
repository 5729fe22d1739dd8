"""The version string, part of the key under which launch shapes are kept,
names the sources the kernels were built from."""
import os
import shutil

import paper_0904_0642_gb300 as su3
from paper_0904_0642_gb300 import build, tuning


def test_version_names_the_sources():
    assert f"build {build.build_id()})" in su3.su3_version()


def test_any_source_changes_the_key(tmp_path):
    header = os.path.join(build.HERE, "..", "include", "su3.h")
    csrc = tmp_path / "csrc"
    shutil.copytree(build.CSRC, csrc)
    assert build.build_id(str(csrc), header) == build.build_id()
    cfg, seen = su3.make_config([8, 8, 8, 8]), set()
    for name in sorted(os.listdir(csrc)):
        with open(csrc / name, "a") as f:
            f.write("\n// another line\n")
        seen.add(tuning.key_of([cfg], f"su3gb300 ({build.build_id(str(csrc), header)})"))
    seen.add(tuning.key_of([cfg], f"su3gb300 ({build.build_id()})"))
    assert len(seen) == len(os.listdir(csrc)) + 1
