"""The calls that a layer makes go through a small extension: it passes what ctypes would pass, and what ctypes refuses stays
refused.  No device is needed: a stand-in library records what it is given."""
import ctypes as C
import shutil
import subprocess
import threading
import types

import numpy as np
import pytest
import torch

from paper_2409_15355_b200 import binding as B

STREAM = types.SimpleNamespace(cuda_stream=0x5000)
I32 = [11, -12, 2 ** 31 - 1, -2 ** 31, 15, 16]


def _calls(seg, pages, tensor, numbers, ctx=None):
    """Every hot call of the binding with `tensor()` for each tensor and `numbers()` for each count."""
    t, n = tensor, numbers
    return {
        "ba_reencode_k": lambda: B.ba_reencode_k(ctx, t(), t(), n(), t(), t(), t(), n(), n(), STREAM),
        "ba_reencode_k_paged": lambda: B.ba_reencode_k_paged(ctx, t(), pages, t(), t(), t(), n(), n(), STREAM),
        "ba_block_prefill": lambda: B.ba_block_prefill(ctx, t(), t(), t(), t(), t(), seg, n(), n(), STREAM),
        "ba_block_prefill_bwd": lambda: B.ba_block_prefill_bwd(ctx, t(), t(), t(), t(), t(), t(), t(), t(), t(), seg, n(), n(), STREAM),
        "ba_final_attend": lambda: B.ba_final_attend(ctx, t(), t(), t(), n(), t(), t(), n(), t(), n(), t(), t(), seg, n(), n(), STREAM),
        "ba_final_attend_fused": lambda: B.ba_final_attend_fused(ctx, t(), t(), t(), n(), t(), t(), n(), t(), n(), t(), t(), seg, n(), n(),
                                                                 STREAM, k_out=t()),
        "ba_final_attend_paged": lambda: B.ba_final_attend_paged(ctx, t(), t(), t(), n(), t(), n(), t(), pages, t(), t(), seg, n(), n(), STREAM),
        "ba_final_attend_fused_paged": lambda: B.ba_final_attend_fused_paged(ctx, t(), t(), t(), n(), t(), t(), pages, n(), t(), t(), seg, n(),
                                                                             n(), STREAM, k_out=t()),
        "ba_segment": lambda: B.ba_segment(ctx, t(), t(), n(), n(), n(), n(), torch.zeros(48, dtype=torch.uint8), STREAM),
    }


NAMES = sorted(_calls(None, None, None, None))


@pytest.fixture()
def recorder(tmp_path):
    """A library with the prototypes of the hot calls that keeps every argument (of a structure: its first words)."""
    lib = B.load_library()
    if shutil.which("gcc") is None or isinstance(B._calls(), B._CtypesCalls):
        pytest.skip("no C compiler")
    src = ["#include <string.h>", "long long rec[64]; int n_rec;", "#define A(x) rec[n_rec++] = (long long)(x);"]
    for name in NAMES:
        types_ = getattr(lib, name).argtypes
        kinds = ["int" if t in (C.c_int32, C.c_int) else "unsigned long" if t is C.c_size_t else "void *" for t in types_]
        body = "".join(f"A(a{i})" if not issubclass(t, C._Pointer) or name == "ba_segment" else
                       f"A(((int *)a{i})[0]) A(((int *)a{i})[1]) A(((long long *)a{i})[1])" for i, t in enumerate(types_))
        src.append(f"int {name}({', '.join(f'{k} a{i}' for i, k in enumerate(kinds))}) {{ n_rec = 0; {body} return 0; }}")
    c, so = tmp_path / "rec.c", tmp_path / "rec.so"
    c.write_text("\n".join(src))
    subprocess.run(["gcc", "-shared", "-fPIC", str(c), "-o", str(so)], check=True)
    fake = C.CDLL(str(so))
    for name in NAMES:
        getattr(fake, name).argtypes = getattr(lib, name).argtypes
    rec, n_rec = (C.c_longlong * 64).in_dll(fake, "rec"), C.c_int.in_dll(fake, "n_rec")
    marshal = B._calls()
    marshal.bind(fake._handle, None, C.c_void_p, B.ba_segments, B.ba_page_table)
    yield fake, lambda: list(rec)[:n_rec.value]
    marshal.bind(lib._handle, B._through_ctypes, C.c_void_p, B.ba_segments, B.ba_page_table)


@pytest.mark.parametrize("name", NAMES)
@pytest.mark.parametrize("ctx", [None, C.c_void_p(0x7000), 0x7100], ids=["null", "handle", "int"])
def test_the_extension_passes_what_ctypes_passes(recorder, name, ctx, monkeypatch):
    fake, given = recorder
    seg, pages = B.ba_segments(batch=3, n_blocks=4, n_tokens=5), B.ba_page_table(64, 7, 0x9000, 0xa000)
    tensors = [torch.zeros(8), 0x1234567890, None, torch.zeros(2, 3, dtype=torch.bfloat16), 2 ** 64 - 16, 0, torch.zeros(0)]

    def fresh():
        it, nt = iter(tensors * 3), iter(I32 * 2)
        return (lambda: next(it)), (lambda: next(nt))
    t, n = fresh()
    _calls(seg, pages, t, n, ctx)[name]()
    fast = given()
    t, n = fresh()
    monkeypatch.setattr(B, "_lib", fake)                     # the other way, asked for directly
    way = types.SimpleNamespace(**{k[3:]: (lambda *a, k=k: B._through_ctypes(k, *a)) for k in NAMES})
    monkeypatch.setattr(B, "_marshal", way)
    _calls(seg, pages, t, n, ctx)[name]()
    slow = given()
    if name == "ba_segment":                                  # (each call has a structure and a buffer of its own)
        drop = {7, 9}
        fast, slow = ([v for i, v in enumerate(x) if i not in drop] for x in (fast, slow))
    assert fast == slow and len(fast) >= 9


BAD_STRUCTURES = [B.ba_page_table(), np.int32(3), b"abc", None, np.zeros(400, dtype=np.uint8), B.ba_config(), 5, "segments"]


@pytest.mark.parametrize("seg", BAD_STRUCTURES, ids=lambda v: type(v).__name__)
@pytest.mark.parametrize("name", [n for n in NAMES if n not in ("ba_reencode_k", "ba_reencode_k_paged", "ba_segment")])
def test_only_segments_are_taken_as_segments(name, seg):
    with pytest.raises((TypeError, C.ArgumentError)):
        _calls(seg, B.ba_page_table(), lambda: None, lambda: 0)[name]()


@pytest.mark.parametrize("pages", [B.ba_segments(), np.int32(3), b"abc", None, np.zeros(400, dtype=np.uint8), 5], ids=lambda v: type(v).__name__)
@pytest.mark.parametrize("name", [n for n in NAMES if n.endswith("_paged")])
def test_only_page_tables_are_taken_as_page_tables(name, pages):
    with pytest.raises((TypeError, C.ArgumentError)):
        _calls(B.ba_segments(), pages, lambda: None, lambda: 0)[name]()


@pytest.mark.parametrize("bad,error", [(np.int64(0x1000), AttributeError), (b"abcdefgh", AttributeError), (bytearray(16), AttributeError),
                                       (C.c_void_p(16), AttributeError), (memoryview(b"abcdefgh"), AttributeError), (1.5, AttributeError),
                                       (torch.zeros(4, 4).t()[1:], ValueError), ([1, 2], AttributeError)],
                         ids=lambda v: type(v).__name__)
@pytest.mark.parametrize("name", NAMES)
def test_objects_that_are_no_tensors_are_refused(name, bad, error):
    with pytest.raises(error):
        _calls(B.ba_segments(), B.ba_page_table(), lambda: bad, lambda: 0)[name]()


@pytest.mark.parametrize("bad", [1.5, "7", None, np.float32(2)], ids=lambda v: type(v).__name__)
@pytest.mark.parametrize("name", NAMES)
def test_numbers_are_taken_as_ctypes_takes_them(name, bad):
    with pytest.raises((TypeError, C.ArgumentError)):
        _calls(B.ba_segments(), B.ba_page_table(), lambda: None, lambda: bad)[name]()


@pytest.mark.parametrize("number", [C.c_int32(0), True, 2 ** 40, np.int64(3)], ids=["c_int32", "bool", "wide", "int64"])
@pytest.mark.parametrize("name", NAMES)
def test_calls_without_a_context_reach_the_library(name, number):
    """Arguments the library itself refuses (no context), numbers in every form ctypes takes, host arrays by their address."""
    with pytest.raises(B.BaError) as e:
        _calls(B.ba_segments(), B.ba_page_table(page_rows=16), lambda: np.zeros(8, dtype=np.int32), lambda: number)[name]()
    assert e.value.status in (B.BA_ERR_INVALID_ARG, B.BA_ERR_UNSUPPORTED)


def test_no_thread_sees_the_extension_before_it_is_bound(monkeypatch):
    """A second thread's first call while one loads the library: it waits for what is complete."""
    seen, bound = [], []

    class Extension:
        def bind(self, *args):
            other = threading.Thread(target=lambda: seen.append((B._calls(), list(bound))))
            other.start()
            other.join(0.3)
            bound.append(1)
            self.other = other
    e = Extension()
    for name, value in (("_lib", None), ("_marshal", None), ("_load_marshal", lambda: e)):
        monkeypatch.setattr(B, name, value)
    B.load_library()
    e.other.join()
    assert seen == [(e, [1])]
