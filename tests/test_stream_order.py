"""A solve's work on its two streams: what a kernel reads has been written before it, by
the order of a stream, an event or a host synchronisation, whatever the timing; and every
launch is counted once.  The host code runs against a CUDA runtime without a device that
writes the calls down (fake_cudart.c)."""
import ctypes
import glob
import os
import subprocess

import numpy as np
import pytest

from paper_2210_07021_gb300 import build, sfmm

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    sfmm.load()
    objects = [os.path.join(build.OUT, f.replace(".cu", ".o")) for f in build.sources()]
    if not all(map(os.path.exists, objects)):
        build.build(force=True)
    tmp = str(tmp_path_factory.mktemp("fake"))
    subprocess.run(["gcc", "-O1", "-fPIC", "-c", os.path.join(HERE, "fake_cudart.c"), "-o", tmp + "/fake.o"], check=True)
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", tmp + "/lib.so", *objects, tmp + "/fake.o"], check=True)
    L = ctypes.CDLL(tmp + "/lib.so")
    L.fake_trace.restype = ctypes.c_char_p
    return L


def trace(lib, call, precision, **options):
    """[(kernel or operation, the operations that are done before it)] of one call, and its launch count."""
    o = sfmm.Options()
    lib.sfmm_default_options(ctypes.byref(o))
    o.precision = precision
    for k, v in options.items():
        setattr(o, k, v)
    h = ctypes.c_void_p()
    lib.sfmm_plan(ctypes.byref(h), 29, 8, ctypes.c_double(0), ctypes.byref(o))
    a = [np.zeros(8192) for _ in range(7)]
    p = [ctypes.c_void_p(x.ctypes.data) for x in a]
    n = ctypes.c_int64(100)
    lib.fake_clear()
    if call == "adjoint":
        st = lib.sfmm_adjoint(h, p[0], p[1], n, p[2], n, p[3], p[4], p[5], p[6])
    elif call == "shear":
        st = lib.sfmm_shear(h, p[0], p[1], n, p[2], n, None, None, p[3], None)
    else:
        st = getattr(lib, call)(h, p[0], p[1], n, p[2], n, p[3], p[4])
    assert st == sfmm.SFMM_OK
    done, event, host, ops = {}, {}, 0, []      # sets of operations as bits
    for line in lib.fake_trace().decode().splitlines():
        what, s, *more = line.split()
        before = done.get(s, 0) | host
        if what == "record":
            event[more[0]] = before
        elif what == "wait":
            done[s] = before | event.get(more[0], 0)
        elif what == "sync":
            host |= before
        else:
            done[s] = before | 1 << len(ops)
            ops.append((more[0] if what == "launch" else what, before))
    stats = sfmm.Stats()
    lib.sfmm_get_stats(h, ctypes.byref(stats))
    lib.sfmm_destroy(h)
    return ops, stats.launches


# what the near-field kernel of each path reads, beside the lists and the targets
NEAR = {sfmm.SFMM_FP64: ("k_eval", ["k_gather_src", "k_p2m64_leaf"]),
        sfmm.SFMM_MIXED: ("k_eval32", ["k_src_offsets", "k_tgt_offsets"]),
        sfmm.SFMM_MIXED_DF: ("k_eval_df", ["k_src_offsets", "k_tgt_offsets"]),
        sfmm.SFMM_FP32: ("k_eval32", ["k_src_offsets", "k_tgt_offsets"])}


@pytest.mark.parametrize("precision", sorted(NEAR))
@pytest.mark.parametrize("call", ["sfmm_deflection", "sfmm_deflection_host", "shear", "adjoint"])
def test_near_field_comes_after_what_it_reads(lib, call, precision):
    near, written = NEAR[precision]
    if call == "shear":
        near, written = NEAR[sfmm.SFMM_FP64]
    elif call == "adjoint":
        near, written = NEAR[sfmm.SFMM_MIXED_DF] if precision != sfmm.SFMM_FP64 else ("k_eval_adj", ["k_gather_dip", "k_p2m_adj"])
    ops, _ = trace(lib, call, precision)
    is_ = lambda name, k: f"{len(k)}{k}" in name        # a mangled name holds its length
    reads = [i for i, (name, _) in enumerate(ops) if is_(name, near)]
    assert reads
    for k in written + ["k_gather_tgt", "k_collect", "k_walk_round", "k_csr_offsets"]:
        at = [i for i, (name, _) in enumerate(ops[:reads[0]]) if is_(name, k)]
        assert at, k
        for i in at:
            assert ops[reads[0]][1] >> i & 1, f"{near} does not wait for {k}"
    # M2L comes after the lists, and the call's last operation after everything before it
    walk = [i for i, (name, _) in enumerate(ops) if is_(name, "k_walk_round")]
    for name, before in ops:
        if "k_m2l" in name or "k_pair_geo" in name:
            assert all(before >> i & 1 for i in walk)
    assert ops[-1][1] == (1 << len(ops) - 1) - 1


COUNTED = [(call, precision, options) for precision in sorted(NEAR)
           for call in ("sfmm_deflection", "sfmm_deflection_host", "shear")
           for options in ({}, {"m2l_tensor_cores": 0})]
COUNTED += [(call, sfmm.SFMM_FP64, {"sigma": 0.1}) for call in ("sfmm_deflection", "sfmm_deflection_host")]


@pytest.mark.parametrize("call,precision,options", COUNTED)
def test_every_launch_is_counted_once(lib, call, precision, options):
    ops, launches = trace(lib, call, precision, **options)
    assert launches == sum(name.startswith("_Z") for name, _ in ops)
