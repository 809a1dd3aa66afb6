"""Error words of the device on the library's host side (no GPU needed): fastpc_api.cu compiled for
the CPU against a fake of the CUDA runtime and of the launchers (fake_cuda.cpp), whose device
memory holds anything and whose products report expired waits on demand.  An error
reaches the call that returns what it spoilt, whatever the order of the calls, and goes with
the data that it belongs to."""
import ctypes
import importlib.util
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2109_04626_gb300")
TIMEOUT = 7


@pytest.fixture(scope="module")
def fp(tmp_path_factory):
    cuda = "/usr/local/cuda/include"
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are missing")
    d = tmp_path_factory.mktemp("host")
    flags = ["g++", "-std=c++17", "-O1", "-fPIC", "-I", cuda, "-I", os.path.join(PKG, "csrc"),
             "-I", os.path.join(ROOT, "include")]
    objs = []
    for src in (os.path.join(PKG, "csrc", "fastpc_api.cu"), os.path.join(ROOT, "tests", "fake_cuda.cpp")):
        objs.append(str(d / (os.path.basename(src) + ".o")))
        subprocess.run(flags + ["-x", "c++", "-c", src, "-o", objs[-1]], check=True, timeout=300)
    # what no test here needs: an unknown CUDA error
    names = [ln.split() for o in objs for ln in
             subprocess.run(["nm", o], check=True, capture_output=True, text=True).stdout.splitlines()]
    missing = {f[-1] for f in names if f[-2] == "U"} - {f[-1] for f in names if f[-2] != "U"}
    stubs = sorted(m for m in missing if m.startswith(("_ZN3fpc", "cuda")))
    (d / "stubs.c").write_text("".join(f"int {m}(void) {{ return 999; }}\n" for m in stubs))
    lib = str(d / "libhost.so")
    # (-Bsymbolic: its own fakes, also beside a CUDA runtime that the process has loaded)
    subprocess.run(["gcc", "-fPIC", "-c", str(d / "stubs.c"), "-o", str(d / "stubs.o")], check=True, timeout=60)
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", lib] + objs + [str(d / "stubs.o")], check=True, timeout=60)
    spec = importlib.util.spec_from_file_location("fastpc_host", os.path.join(PKG, "fastpc.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    mod.LIB_PATH = lib
    mod.fail = lambda exact=0, split=0: mod.load().fake_fail(exact, split)
    yield mod
    mod.fail()


X = [np.zeros((40, p)) for p in (6, 9, 5)]
LARGE = [np.zeros((40, p)) for p in (520, 530)]          # instances above the exact product's size in a batch


def _batch(fp, Xs, **opts):
    return fp.PCBatch([x.shape[0] for x in Xs], [x.shape[1] for x in Xs], 0.01, -1, **opts)


@pytest.mark.parametrize("Xs", [X, LARGE])
@pytest.mark.parametrize("precision", [0, 2])
def test_instances_in_any_order(fp, Xs, precision):
    """The words start clean: no instance has to come first."""
    with _batch(fp, Xs, precision=precision) as pb:
        for i in reversed(range(len(Xs))):
            pb.corr_block(i, Xs[i])
        C32, C64 = pb.corr_get()
        assert np.isfinite(C64).all() and np.isfinite(C32).all()


@pytest.mark.parametrize("Xs", [X, LARGE])
@pytest.mark.parametrize("first", [0, 1])
def test_error_of_one_instance(fp, Xs, first):
    """An instance's expired wait is reported until that instance is given again, and by no other order."""
    with _batch(fp, Xs) as pb:
        order = [1, 0, 2][:len(Xs)]
        fp.fail(1, 1)
        for i in (order if first else order[::-1]):
            pb.corr_block(i, Xs[i])
        fp.fail()
        bad = (order if first else order[::-1])[0]
        for _ in range(2):
            with pytest.raises(fp.PCError) as e:
                pb.corr_get()
            assert e.value.status == TIMEOUT
            other = 0 if bad else 1
            pb.corr_block(other, Xs[other])               # a good instance again changes nothing
        pb.corr_block(bad, Xs[bad])
        pb.corr_get()


@pytest.mark.parametrize("Xs", [X, LARGE])
def test_error_in_one_call_for_all(fp, Xs):
    with _batch(fp, Xs) as pb:
        fp.fail(2, 2)
        pb.corr_blocks(Xs)
        with pytest.raises(fp.PCError) as e:
            pb.corr_get()
        assert e.value.status == TIMEOUT
        pb.corr_blocks(Xs)
        pb.corr_get()


def _raw(fp, h, l):
    """One raw test; its r."""
    ij, S, r = np.zeros(2, np.int32), np.zeros(max(l, 1), np.int32), np.zeros(1)
    fp._check(h, fp.load().pc_ci_batch(h, ij.ctypes.data, S.ctypes.data, l, 1, r.ctypes.data, None, None))
    return r[0]


def _features(fp, h, l):
    q, f = np.zeros(4, np.int32), np.zeros(16, np.float32)
    fp._check(h, fp.load().pc_mlp_features(h, q.ctypes.data, 1, f.ctypes.data))


@pytest.mark.parametrize("call", [_raw, _features])
@pytest.mark.parametrize("p, opts", [(20, {}), (20, dict(order=0)), (150, dict(order=0)), (150, {}), (20, dict(precision=0))])
def test_values_of_a_failed_product_are_refused(fp, call, p, opts):
    with fp.PC(40, p, 0.01, **opts) as pc:
        fp.fail(1, 1)
        pc.corr(np.zeros((40, p)))
        fp.fail()
        for l in (4, 0):
            with pytest.raises(fp.PCError) as e:
                call(fp, pc.h, l)
            assert e.value.status == TIMEOUT
        pc.corr(np.zeros((40, p)))
        for l in (0, 4):
            call(fp, pc.h, l)


def test_raw_tests_need_no_work_put_off(fp):
    """Everything a raw test reads is formed by pc_corr: the caller's data are not needed later."""
    with fp.PC(40, 20, 0.01) as pc:
        for _ in range(2):
            before = fp.load().fake_split()
            pc.corr(np.zeros((40, 20)))
            assert fp.load().fake_split() == before + 1
            assert _raw(fp, pc.h, 0) == 0.5 and _raw(fp, pc.h, 0) == 0.5
            assert fp.load().fake_split() == before + 1


def test_error_of_the_split_product_alone(fp):
    """It spoils the raw tests that read it, not the search, and goes with the next data."""
    with fp.PC(40, 20, 0.01) as pc:
        fp.fail(0, 1)
        pc.corr(np.zeros((40, 20)))
        fp.fail()
        with pytest.raises(fp.PCError) as e:
            _raw(fp, pc.h, 0)
        assert e.value.status == TIMEOUT
        pc.corr_get()
        pc.skeleton()
        pc.corr(np.zeros((40, 20)))
        _raw(fp, pc.h, 0)


def test_device_skeleton_of_a_failed_product(fp):
    """The skeleton of an unfinished matrix does not reach a device output."""
    out = np.full((20, 20), 9, np.uint8)
    fp.load().fake_device(ctypes.c_void_p(out.ctypes.data), ctypes.c_longlong(out.size))
    with fp.PC(40, 20, 0.01) as pc:
        fp.fail(1, 0)
        pc.corr(np.zeros((40, 20)))
        with pytest.raises(fp.PCError) as e:
            pc.skeleton(out)
        assert e.value.status == TIMEOUT
        assert (out == 9).all()
        pc.corr(np.zeros((40, 20)))
        pc.skeleton(out)
        assert (out == 1).all()


@pytest.mark.parametrize("batch", [False, True])
def test_no_search_on_an_unfinished_split_product(fp, batch):
    """Its matrix holds anything where it did not finish, and a search of it can take any time: halted
    on the device before the first stage."""
    with _batch(fp, LARGE, graph=0) if batch else fp.PC(40, 150, 0.01, order=0, graph=0) as pc:
        before = fp.load().fake_halted()
        fp.fail(0, 2 if batch else 1)
        for i, x in enumerate(LARGE) if batch else []:
            pc.corr_block(i, x)
        if not batch:
            pc.corr(np.zeros((40, 150)))
        fp.fail()
        with pytest.raises(fp.PCError) as e:
            pc.skeleton()
        assert e.value.status == TIMEOUT
        assert fp.load().fake_halted() == before + 1
