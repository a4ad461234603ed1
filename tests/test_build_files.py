"""Builds that run at the same time: an object, the library or the stamp is never
seen half-written under its own name.  A stand-in for nvcc writes its output in two
halves; a second thread looks at the files meanwhile."""
import importlib.util
import os
import shutil
import threading

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

NVCC = """#!/bin/sh
while [ $# -gt 0 ]; do
  if [ "$1" = -o ]; then out=$2; fi
  shift
done
printf half > "$out"
sleep 0.3
printf ' and whole' >> "$out"
"""


def test_files_appear_whole(tmp_path, monkeypatch):
    pkg = tmp_path / "paper_1611_03189_gb300"
    shutil.copytree(os.path.join(ROOT, "paper_1611_03189_gb300", "csrc"), pkg / "csrc")
    shutil.copy(os.path.join(ROOT, "paper_1611_03189_gb300", "build.py"), pkg)
    shutil.copytree(os.path.join(ROOT, "include"), tmp_path / "include")
    nvcc = tmp_path / "nvcc"
    nvcc.write_text(NVCC)
    nvcc.chmod(0o755)
    monkeypatch.setenv("NVCC", str(nvcc))
    spec = importlib.util.spec_from_file_location("build_copy", pkg / "build.py")
    B = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(B)
    names = [os.path.join(B.BUILD, s + ".o") for s in B.SOURCES] + [B.LIB]
    seen, done = set(), threading.Event()

    def look():
        while not done.is_set():
            for n in names:
                if os.path.exists(n):
                    with open(n) as f:
                        seen.add(f.read())

    t = threading.Thread(target=look)
    t.start()
    try:
        B.build()
    finally:
        done.set()
        t.join()
    assert seen <= {"half and whole"}
    assert sorted(os.listdir(B.BUILD)) == sorted([os.path.basename(n) for n in names] + ["ARCH"])
