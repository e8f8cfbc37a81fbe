"""The native call of topk(): a module that is missing, damaged or made for another torch leaves the general call, and is built again."""
import os
import shutil
import subprocess

import pytest
import torch

from paper_2106_05203_b200 import binding, build


def _changed(path, to):
    """A copy of the module that says it was built for another torch."""
    old = build.call_built_for().encode()
    data = open(binding.CALL_PATH, "rb").read()
    assert data.count(old) >= 1
    open(path, "wb").write(data.replace(old, to.ljust(len(old))[:len(old)].encode()))


@pytest.mark.parametrize("kind", ["missing", "damaged", "another torch", "another module"])
def test_the_general_call_is_left(kind, tmp_path):
    path = str(tmp_path / "_topk_call.so")
    if kind == "damaged":
        open(path, "wb").write(b"no shared object")
    elif kind == "another torch":
        _changed(path, "torch 1.0")
    elif kind == "another module":
        shutil.copy(binding.LIB_PATH, path)                    # no module at all
    with pytest.warns(RuntimeWarning, match="without its native call"):
        call = binding._load_call(path)
    assert call(torch.zeros(4), 1) is None


def test_the_module_that_fits_is_taken(recwarn):
    assert binding._load_call() is not None and not [w for w in recwarn if "native call" in str(w.message)]


def test_a_module_for_another_torch_is_built_again(tmp_path, monkeypatch):
    path, commands = str(tmp_path / "_topk_call.so"), []

    def run(command, check):
        commands.append(command)
        open(command[command.index("-o") + 1], "w").close()
    monkeypatch.setattr(build, "CALL", path)
    monkeypatch.setattr(subprocess, "run", run)
    shutil.copy(binding.CALL_PATH, path)
    os.utime(path)
    build.build_call()
    assert commands == []
    _changed(path, "torch 1.0")
    build.build_call()
    assert len(commands) == 1
