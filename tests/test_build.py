"""The shared objects appear whole, whatever else loads or builds them, and stay valid where a tree is copied to."""
import os
import shutil
import subprocess
import sys
import threading

import pytest

from paper_2409_15355_b200 import build as b

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_output_is_replaced_whole(tmp_path):
    """A compiler that writes its output in two halves, two builds at a time: a reader never sees half a file."""
    out, cc = tmp_path / "lib.so", tmp_path / "cc.py"
    cc.write_text("import sys, time\nf = open(sys.argv[sys.argv.index('-o') + 1], 'w')\nf.write('a' * 1000)\nf.flush()\ntime.sleep(.2)\n"
                  "f.write('b' * 1000)\nf.close()\n")
    out.write_text("o" * 2000)
    held = open(out)                                          # a process that has the old file open keeps it
    errors, seen, done = [], set(), threading.Event()

    def one():
        try:
            for _ in range(2):
                b._compile([sys.executable, str(cc)], str(out), "digest", "failed:\n")
        except Exception as e:                                # noqa: BLE001
            errors.append(e)
    threads = [threading.Thread(target=one) for _ in range(2)]
    reader = threading.Thread(target=lambda: [seen.add(out.read_text()) for _ in iter(done.is_set, True)])
    reader.start()
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    done.set(); reader.join()
    assert not errors and seen <= {"o" * 2000, "a" * 1000 + "b" * 1000} and held.read() == "o" * 2000
    assert (tmp_path / "lib.so.hash").read_text() == "digest" and sorted(os.listdir(tmp_path)) == ["cc.py", "lib.so", "lib.so.hash"]


def test_a_failed_build_leaves_the_old_file(tmp_path):
    out = tmp_path / "lib.so"
    out.write_text("old")
    with pytest.raises(RuntimeError, match="no good: "):
        b._compile([sys.executable, "-c", "import sys; sys.exit('sources')"], str(out), "digest", "no good: ")
    assert out.read_text() == "old" and os.listdir(tmp_path) == ["lib.so"]


def test_a_copied_tree_keeps_its_builds(tmp_path):
    b.build(); b.build_marshal()
    for d in ("paper_2409_15355_b200", "include"):
        shutil.copytree(os.path.join(ROOT, d), tmp_path / d)
    code = "from paper_2409_15355_b200 import build as b; print(b.build(), b.build_marshal())"
    env = dict(os.environ, NVCC="/nonexistent/nvcc", CC="/nonexistent/cc", PYTHONPATH=str(tmp_path))
    got = subprocess.run([sys.executable, "-c", code], cwd=tmp_path, env=env, capture_output=True, text=True)
    assert got.returncode == 0, got.stderr
    assert got.stdout.split() == [str(tmp_path / "paper_2409_15355_b200" / n) for n in ("libba.so", "ba_marshal.so")]


@pytest.mark.parametrize("found", ["no_build", "stale_build"])
def test_a_prebuilt_library_loads_without_a_compiler(tmp_path, found):
    """BA_LIBRARY names a library to use as it is: neither a compiler nor a writable folder is needed beside it."""
    lib = b.build()
    for d in ("paper_2409_15355_b200", "include"):
        shutil.copytree(os.path.join(ROOT, d), tmp_path / d, ignore=shutil.ignore_patterns("*.so", "*.hash", "__pycache__"))
    if found == "stale_build":
        (tmp_path / "paper_2409_15355_b200" / "ba_marshal.so").write_text("of other sources")
        (tmp_path / "paper_2409_15355_b200" / "ba_marshal.so.hash").write_text("of other sources")
    code = ("import types, warnings\nfrom paper_2409_15355_b200 import binding as B\n"
            "with warnings.catch_warnings(record=True) as w:\n    warnings.simplefilter('always')\n    B.load_library()\n"
            "assert [x.category for x in w if x.category is not ResourceWarning] == [RuntimeWarning], [str(x) for x in w]\n"
            "s = types.SimpleNamespace(cuda_stream=0)\n"
            "try:\n    B.ba_block_prefill(None, None, None, None, None, None, B.ba_segments(), 0, 0, s)\n"
            "except B.BaError as e:\n    assert e.status == B.BA_ERR_INVALID_ARG\n"
            "else:\n    raise SystemExit('no error')\n"
            "try:\n    B.ba_block_prefill(None, None, None, None, None, None, None, 0, 0, s)\n"
            "except TypeError:\n    print('loaded')\n")
    env = dict(os.environ, NVCC="/nonexistent/nvcc", CC="/nonexistent/cc", PYTHONPATH=str(tmp_path), BA_LIBRARY=lib)
    got = subprocess.run([sys.executable, "-c", code], cwd=tmp_path, env=env, capture_output=True, text=True)
    assert got.returncode == 0 and got.stdout.strip() == "loaded", got.stderr
