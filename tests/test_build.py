"""When the extension _pf_ext is compiled again: its sources, and the torch and Python that it was built against."""
import os

import torch

from paper_2504_00492_b200 import build


def test_the_extension_is_rebuilt_for_another_torch(monkeypatch, tmp_path):
    runs = []

    def compiler(cmd, check):
        runs.append(cmd)
        with open(cmd[cmd.index("-o") + 1], "w") as f:
            f.write("built")

    monkeypatch.setattr(build, "EXT", str(tmp_path / "_pf_ext.so"))
    monkeypatch.setattr(build, "EXT_TAG", str(tmp_path / "sub" / "tag"), raising=False)
    monkeypatch.setattr(build.subprocess, "run", compiler)
    build.build_ext()
    build.build_ext()
    assert len(runs) == 1                                   # up to date
    monkeypatch.setattr(torch, "__version__", "99.0")
    build.build_ext()
    build.build_ext()
    assert len(runs) == 2                                   # another torch, its sources' dates notwithstanding
    os.utime(build.EXT, (1, 1))
    build.build_ext()
    assert len(runs) == 3                                   # older than its sources
