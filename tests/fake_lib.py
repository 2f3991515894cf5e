"""A copy of the package whose library is compiled with fake_cuda.h in front of every source, for
what a working GPU does not let happen. Scripts run against it in a process of their own."""
import importlib.util
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
PACKAGE = "paper_1907_12343_gb300"


_built = None


def build(tmp_path_factory) -> str:
    """Copy and compile, once per process; returns the directory to import the package from."""
    global _built
    if _built is None:
        _built = _build(str(tmp_path_factory.mktemp("fake")))
    return _built


def _build(where: str) -> str:
    shutil.copytree(os.path.join(ROOT, "include"), os.path.join(where, "include"))
    shutil.copytree(os.path.join(ROOT, PACKAGE), os.path.join(where, PACKAGE),
                    ignore=shutil.ignore_patterns("_build", "__pycache__"))
    spec = importlib.util.spec_from_file_location("_fake_build", os.path.join(where, PACKAGE, "build.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    mod.build(force=True, extra_flags=("-include", os.path.join(HERE, "fake_cuda.h")))
    return where


def run(where, script, timeout=300) -> str:
    """Run a script with the copied package first on the path (then this repository's modules)."""
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([where, HERE, ROOT]))
    res = subprocess.run([sys.executable, "-c", script], capture_output=True, text=True, timeout=timeout, env=env, cwd=where)
    assert res.returncode == 0, res.stdout + res.stderr
    return res.stdout
