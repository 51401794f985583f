"""The build entry point on a tree without a built library, as a fresh checkout is."""
import os
import shutil
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PACKAGE = "paper_2502_06352_b200"


def test_build_needs_no_library_to_start_from(tmp_path):
    tree = tmp_path / "tree"
    shutil.copytree(os.path.join(ROOT, PACKAGE), tree / PACKAGE, ignore=shutil.ignore_patterns("*.so", "_build", "__pycache__"))
    shutil.copytree(os.path.join(ROOT, "include"), tree / "include")
    shutil.copy(os.path.join(ROOT, "__graft_entry__.py"), tree)
    # in the compiler's place: an object file is an empty file, the linked library the one that is built already
    nvcc = tmp_path / "nvcc"
    nvcc.write_text('#!/bin/sh\nout=; shared=0\nwhile [ $# -gt 0 ]; do case "$1" in -o) shift; out="$1";; -shared) shared=1;; esac; shift; done\n'
                    'if [ $shared = 1 ]; then cp "%s" "$out"; else : > "$out"; fi\n' % os.path.join(ROOT, PACKAGE, "liblantern.so"))
    nvcc.chmod(0o755)
    env = dict(os.environ, NVCC=str(nvcc))
    env.pop("PYTHONPATH", None)
    r = subprocess.run([sys.executable, "-c", "import __graft_entry__ as g; g.build()"], cwd=tree, env=env,
                       stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:]
    assert (tree / PACKAGE / "liblantern.so").exists()
