"""The C ABI library loads and exports every function include/*.h declares
(no GPU needed: nothing is launched)."""
import ctypes
import glob
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_functions():
    names = set()
    for h in glob.glob(os.path.join(ROOT, "include", "*.h")):
        src = open(h).read()
        src = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
        for m in re.finditer(r"^\s*(?:const\s+)?[A-Za-z_][\w\s\*]*?\b(fn_\w+)\s*\(", src, flags=re.M):
            names.add(m.group(1))
    return sorted(names)


def test_header_declares_entry_points():
    names = declared_functions()
    for must in ("fn_time_edges", "fn_knn_tree", "fn_rnea_dump", "fn_status_str"):
        assert must in names


def test_library_exports_declared_symbols():
    from paper_2609_22608_gb300 import _build
    _build.build()
    lib = ctypes.CDLL(_build.LIB)
    missing = [n for n in declared_functions() if not hasattr(lib, n)]
    assert not missing, missing
    lib.fn_status_str.restype = ctypes.c_char_p
    assert lib.fn_status_str(-1).startswith(b"FN_EINVAL")


def test_oracle_builds_and_is_separate():
    import oracle
    oracle.build()
    # the oracle and the CUDA path share no sources
    csrc = os.path.join(ROOT, "paper_2609_22608_gb300", "csrc")
    for f in glob.glob(os.path.join(csrc, "*")):
        assert "fn_oracle" not in open(f).read()
    for f in glob.glob(os.path.join(ROOT, "oracle", "*.[ch]")):
        text = open(f).read()
        assert "fn_api.h" not in text and "csrc" not in text


@pytest.mark.parametrize("form", ["float32", "float64", "lists", "item"])
def test_arm_struct_forms(form):
    """The block conversion of an arm dict fills the struct as the item-wise
    one does, whatever holds the values, and raises its errors."""
    from paper_2609_22608_gb300 import _lib, synth
    for seed in range(3):
        arm = synth.make_arm(seed)
        if form == "float64":
            arm = {k: np.asarray(v, np.float64) if k != "dof" else v for k, v in arm.items()}
        elif form == "lists":
            arm = {k: np.asarray(v).tolist() for k, v in arm.items()}
        elif form == "item":              # a shape that only item assignment takes
            arm = dict(arm, com=np.vstack([arm["com"], arm["com"][:1]]))
        assert bytes(_lib.arm_struct(arm)) == bytes(_lib._arm_struct_by_item(arm))
    with pytest.raises(ValueError):
        _lib.arm_struct(dict(synth.make_arm(0), dh_a=np.zeros(5, np.float32)))


def test_knn_workspace_bound():
    """The workspace of the parent search stays within what the header states, for
    few and many queries on small and large trees."""
    from paper_2609_22608_gb300 import ops
    for N in (1, 255, 256, 257, 2047, 2048, 2049, 4096, 65536, 131073, 10 ** 6, 2799999, 3 * 10 ** 6):
        for B in (1, 255, 257, 8192, 65536, 200000, 262144, 10 ** 6):
            for k in (1, 8, 16):
                nodes = (N + 127) // 128 * 128
                batch = max(88 << 20, (24 << 10) + 32 * (nodes + 2048) if N >= 2800000 else 0)
                need = ops.knn_workspace_bytes(B, N, k)
                assert need <= batch + 256 + 152 * nodes, (B, N, k, need)
                assert N < 256 or need >= 152 * nodes + 1024
    # the largest planner's search is one batch: 8192 queries' minima of 65536 nodes
    assert ops.knn_workspace_bytes(8192, 65536, 16) >= 8192 * 8192 + 152 * 65536


def test_arm_struct_scalars():
    """Scalar fields may be anything that float() takes, as in the item-wise
    conversion, and dof any integer that a C int holds in its way."""
    import torch

    from paper_2609_22608_gb300 import _lib, synth
    arm = synth.make_arm(1)
    arm = dict(arm, w_max=torch.tensor(float(arm["w_max"]), requires_grad=True),
               blade_len=str(float(arm["blade_len"])), flange_d=np.float64(arm["flange_d"]))
    assert bytes(_lib.arm_struct(arm)) == bytes(_lib._arm_struct_by_item(arm))
    arm["dof"] = 2 ** 32 + 7
    assert _lib.arm_struct(arm).dof == 7
    with pytest.raises((TypeError, ValueError)):
        _lib.arm_struct(dict(arm, w_max="wide"))
