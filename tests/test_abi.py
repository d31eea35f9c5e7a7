"""CPU-side checks of the C-ABI library: it loads without a GPU, exports every symbol the
header declares, and rejects bad arguments on the host before anything is launched."""
import ctypes
import os
import re

import pytest

import paper_2608_20427_b200 as bf1
from paper_2608_20427_b200 import binding

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_functions():
    text = open(os.path.join(ROOT, "include", "bf1.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(bf1_[a-z0-9_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported():
    lib = bf1.load()
    names = declared_functions()
    assert set(binding.EXPORTS) <= set(names)
    for name in names:
        assert hasattr(lib, name), name
    assert lib.bf1_version() >= 1


def test_route_capacity_is_host_only_and_matches_the_degree_bound():
    cap, deg = bf1.route_capacity(1, 32768, 32768)
    assert cap >= 512 and deg == 11          # floor(log2 511) + 3
    cap, deg = bf1.route_capacity(4, 39922, 16384)
    assert cap >= 47 + 128 + 193 + 256 and deg == 10
    assert bf1.route_capacity(1, 1000, 1000) == (16, 6)
    assert bf1.route_capacity(1, 64, 64)[1] == 1
    assert bf1.route_capacity(1, 257, 257)[1] == 4
    # other routes
    assert bf1.route_capacity(1, 6400, 6400, bf1.RouteCfg(local_blocks=5, global_first=0, dyadic=0))[1] == 6
    assert bf1.route_capacity(1, 6400, 6400, bf1.RouteCfg(local_blocks=0, global_first=1, dyadic=0))[1] == 2


def test_bad_arguments_are_rejected_on_the_host():
    with pytest.raises(bf1.Bf1Error) as e:
        bf1.route_capacity(1, 100, 100, bf1.RouteCfg(block=32))
    assert e.value.code == -2 and "64" in str(e.value)
    with pytest.raises(bf1.Bf1Error):
        bf1.route_capacity(-1, 100, 100)
    with pytest.raises(bf1.Bf1Error):
        bf1.route_capacity(1, 100, 100, bf1.RouteCfg(local_blocks=-1))
    lib = bf1.load()
    # null tensors: refused before any CUDA call
    rc = lib.bf1_dense_causal_fwd(None, None, None, None, 1, 64, 64, 2, 1, 64, 0.0, None, None, None, None)
    assert rc == -1 and b"null" in lib.bf1_last_error()
    rc = lib.bf1_attn_fwd(None, None, None, None, 1, 64, 64, 2, 1, 64, 0.0, None, None, None, None)
    assert rc == -1
    # unsupported geometry (pointers are never dereferenced on this path)
    fake = ctypes.c_void_p(0x1000)
    for hq, hkv, d, code in ((8, 1, 64, -2), (6, 2, 64, -2), (2, 1, 96, -2), (3, 2, 64, -1)):
        rc = lib.bf1_dense_causal_fwd(fake, fake, fake, fake, 1, 64, 64, hq, hkv, d, 0.0, fake, fake, None, None)
        assert rc == code, (hq, hkv, d, lib.bf1_last_error())
    rc = lib.bf1_dense_causal_fwd(ctypes.c_void_p(0x1004), fake, fake, fake, 1, 64, 64, 2, 1, 64, 0.0, fake, fake,
                                  None, None)
    assert rc == -1 and b"aligned" in lib.bf1_last_error()
    # empty batch: OK without touching a device
    rc = lib.bf1_dense_causal_fwd(fake, fake, fake, fake, 0, 0, 0, 2, 1, 64, 0.0, fake, fake, None, None)
    assert rc == 0


@pytest.mark.parametrize("kw", [dict(), dict(local_blocks=0), dict(local_blocks=1), dict(local_blocks=3, global_first=0),
                                dict(local_blocks=4), dict(local_blocks=9, dyadic=0), dict(local_blocks=70)],
                         ids=lambda k: ",".join("%s=%s" % i for i in k.items()) or "paper")
def test_route_capacity_is_the_longest_list(kw):
    """The helper looks at the last three blocks only; powers of two are where the list lengths are not monotone."""
    from oracle import bf1_oracle as O
    longest = 0
    _, count, _, _ = O.route(O.cfg(**kw), 64 * 300)
    for nblk in range(1, 301):
        longest = max(longest, int(count[nblk - 1]))
        assert bf1.route_capacity(1, 64 * nblk, 64 * nblk, bf1.RouteCfg(**kw))[1] == longest, nblk


def test_the_call_path_is_built_for_the_torch_and_python_at_hand(monkeypatch):
    """It is compiled against torch's C++ ABI: with another torch in the same tree the module that is there is not used."""
    import sys

    import torch

    from paper_2608_20427_b200 import build
    path = build.host_path()
    assert torch.__version__ in path and sys.implementation.cache_tag in path
    build.build_host()
    commands = []

    class Done:
        returncode, stdout = 0, ""

    monkeypatch.setattr(build.subprocess, "run", lambda cmd, **kw: commands.append(cmd) or Done)
    monkeypatch.setattr(build.os, "replace", lambda *a: None)
    assert build.build_host() == path and not commands          # fresh
    monkeypatch.setattr(torch, "__version__", "0.0.1+other")
    assert build.build_host() != path and len(commands) == 1


def test_the_call_without_allocation_wants_its_outputs():
    import torch
    q, kv = torch.zeros(64, 2, 64, dtype=torch.bfloat16), torch.zeros(64, 1, 64, dtype=torch.bfloat16)
    cu, lse = torch.tensor([0, 64], dtype=torch.int32), torch.zeros(2, 64)
    for out, l in ((None, lse), (torch.zeros_like(q), None), (None, None)):
        with pytest.raises(TypeError, match="out and lse"):
            bf1.attn_fwd_noalloc(q, kv, kv, cu, 64, out, l)


def test_decode_scratch_is_no_larger_than_what_is_used():
    """Partial results stay on the chip: nothing grows with the batch, its heads or its lists."""
    lib = bf1.load()
    for args in ((1, 16, 8, 11, 128), (0, 2, 1, 1, 64), (65535, 64, 16, 64, 128)):
        assert lib.bf1_decode_workspace_bytes(*args) == 16
    for args in ((-1, 16, 8, 11, 128), (1, 0, 8, 11, 128), (1, 16, 0, 11, 128), (1, 15, 8, 11, 128), (1, 16, 8, 0, 128), (1, 16, 8, 11, 0)):
        assert lib.bf1_decode_workspace_bytes(*args) == -1


def test_decode_refuses_more_kv_heads_than_pairs_of_query_heads_fit_a_grid_dimension():
    """65535 pairs of query heads: with four to a KV head half as many KV heads."""
    lib = bf1.load()
    fake = ctypes.c_void_p(0x1000)
    plan = binding._DecodePlanC(11, 0x1000, 0x1000, 0x1000, 0x1000)
    for group, hkv, code in ((1, 65535, 0), (1, 65536, -2), (2, 65535, 0), (2, 65536, -2), (4, 32767, 0), (4, 32768, -2), (4, 65535, -2)):
        rc = lib.bf1_decode_fwd(fake, fake, fake, 1, fake, 0, group * hkv, hkv, 64, 0.0, ctypes.byref(plan), fake, fake, fake, None)
        assert rc == code, (group, hkv, lib.bf1_last_error())
