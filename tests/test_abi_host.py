"""CPU-only checks of the C-ABI library: it loads, exports every symbol the header declares,
and its host-side logic (validation, size planning, error strings) behaves.  No kernel runs."""
import ctypes
import os
import re

import pytest
import torch

import paper_2602_02180_b200 as still
from paper_2602_02180_b200 import build as still_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    still_build.build_library()
    return still.binding.lib()


def _declared_symbols():
    text = open(os.path.join(ROOT, "include", "still.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(still_[a-z_0-9]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(lib):
    names = _declared_symbols()
    assert "still_hybrid_attn_fwd" in names and "still_hybrid_attn_step" in names
    for n in names:
        assert hasattr(lib, n), f"libstill.so does not export {n}"


def test_validation_and_sizes(lib):
    ok = still.StillParams(2, 32, 8, 128, 64, 64)
    assert still.workspace_bytes(ok, 32768) > 0
    assert still.workspace_bytes(ok, 32768) <= still.workspace_bytes(still.StillParams(2, 32, 8, 128, 64, 16), 32768)
    for bad in [
        still.StillParams(2, 32, 7, 128, 64, 64),      # H % Hkv
        still.StillParams(2, 32, 8, 96, 64, 64),       # head dim
        still.StillParams(2, 32, 8, 128, 48, 16),      # chunk
        still.StillParams(2, 32, 8, 128, 64, 65),      # topk > chunk
        still.StillParams(2, 32, 8, 128, 64, -1),
        still.StillParams(0, 32, 8, 128, 64, 64),
        still.StillParams(2, 32, 8, 128, 64, 64, sm_scale=0.0),
        still.StillParams(2, 32, 8, 64, 64, 64, d_f=128),
    ]:
        assert still.workspace_bytes(bad, 1024) == 0
        assert still.state_bytes(bad, 1024) == 0
    lay = still.state_layout(still.StillParams(1, 4, 2, 64, 64, 16), 1000)
    assert lay["capacity"] == 1024 and lay["total"] == still.state_bytes(still.StillParams(1, 4, 2, 64, 64, 16), 1000)
    order = [lay[k] for k in ("header", "k_cache", "v_cache", "score", "sel_idx", "sel_mask", "S", "z", "scratch", "total")]
    assert order == sorted(order) and all(o % 256 == 0 for o in order)
    with pytest.raises(still.StillError):
        still.state_layout(still.StillParams(1, 4, 3, 64, 64, 16), 1000)


def test_null_and_error_codes_without_a_device(lib):
    c = still.StillParams(1, 2, 2, 64, 64, 16).c()
    rc = lib.still_hybrid_attn_fwd(ctypes.byref(c), 128, None, None, None, None, None, None, None, None, None,
                                   None, None, None, 0, None, 0, None)
    assert rc == -1
    rc = lib.still_hybrid_attn_step(ctypes.byref(c), None, 0, 0, None, None, None, None, None, None, None, None,
                                    None, None)
    assert rc == -1
    assert still.strerror(0) == "ok"
    assert {still.strerror(k) for k in range(-7, 0)}.isdisjoint({"unknown status"})
    assert still.strerror(-99) == "unknown status"


def test_binding_refuses_cpu_tensors(lib):
    p = still.StillParams(1, 2, 2, 64, 64, 16, torch.float32)
    x = torch.zeros(1, 2, 128, 64)
    with pytest.raises(RuntimeError, match="no CPU path"):
        still.hybrid_attn_fwd(p, x, x, x, None, None)
    with pytest.raises(RuntimeError, match="no CPU path"):
        still.hybrid_attn_step(p, None, 0, 0, x[:, :, 0], x[:, :, 0], x[:, :, 0])


def test_dependent_kernels_read_nothing_ahead_of_the_wait():
    # Kernels are made resident while their predecessor runs (programmatic stream serialization): each has to wait before
    # anything else, and no pointer parameter may promise (const restrict) that its memory does not change meanwhile.
    csrc = still_build.CSRC
    seen = 0
    for name in sorted(os.listdir(csrc)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(csrc, name)).read())
        for m in re.finditer(r"__global__[^;{]*?\b(\w+_kernel)\(([^{]*)\)\s*\{", text):
            if m.group(1) == "wait_timeout_selftest_kernel":   # launched by itself, in stream order
                continue
            seen += 1
            assert "__restrict__" not in m.group(2), m.group(1)
            ahead = text[m.end():].split("grid_dep_wait();")[0]
            assert re.fullmatch(r"\s*(extern __shared__[^;]*;\s*)?", ahead), (m.group(1), ahead[:200])
        # (device functions that kernels hand such pointers to are inlined into them)
        assert "__restrict__" not in text, name
    assert seen >= 19


def _csrc(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(still_build.CSRC, name)).read())


def test_a_warp_leaves_a_wait_as_a_whole():
    # A bounded wait can succeed in one lane and run out in another.  Roles of whole warps go on to instructions that take the
    # whole warp (tensor-memory loads, votes, __syncwarp): the softmax warps never leave their loop for one and vote behind it,
    # the scan's vote on every wait.
    softmax = _csrc("still_tc.cu").split("softmax_role(", 1)[1].split("producer_role(", 1)[0]
    head = "for (int k = 0; k < n_mine; ++k) {"
    loop, behind = softmax.split(head)[1].split("wait(bar.pv_done + x, (n_mine - 1) & 1, 9);")
    assert not re.search(r"\b(break|return)\b", loop) and loop.count("wait(bar.") == 3
    assert softmax.count("mbar_wait(") == 1 and re.match(r"\s*if \(__all_sync\(0xffffffffu, ok\)\) \{", behind)
    scan = _csrc("still_la_tc.cu").split("la_fused_kernel(", 1)[1].split("MMA issuer", 1)[-1]
    waits = re.findall(r"if \(ok\) ok = mbar_wait\((?!bar,)[^\n]*\n([^\n]*)", scan)   # (bar: of the issuing warp, see there)
    assert len(waits) == 7 and all("ok = __all_sync(0xffffffffu, ok);" in after for after in waits)


def test_producers_leave_no_load_in_flight():
    # Loads of different ring stages need not land in order, and another role can give up after the producer has armed its last
    # stage: every producer with a ring ends with a wait for all stages that may still be filled, not for the last one, and
    # whether or not it has failed itself.
    drain = _csrc("still_tc_ptx.cuh").split("mbar_drain_ring(", 1)[1].split("}", 1)[0]
    parts = [m.strip() for m in re.search(r"for \(int i = ([^;]*); (i < armed); \+\+i\)\s*mbar_wait_drain\(full \+ ([^,]*), ([^;]*), t0\);", drain).groups()]
    first, more, slot, parity = (m.replace("(uint32_t)", "").replace("/", "//").replace("1u", "1") for m in parts)
    first = re.sub(r"(.*) \? (.*) : (.*)", r"(\2) if (\1) else (\3)", first)
    for n_stages in (1, 2, 4, 5, 11, 12):
        for armed in range(40):
            waited, i = {}, eval(first, {"armed": armed, "n_stages": n_stages})
            while eval(more, {"i": i, "armed": armed}):
                at = {"i": i, "n_stages": n_stages}
                waited[eval(slot, at)] = eval(parity, at)
                i += 1
            last = {k % n_stages: k // n_stages % 2 for k in range(armed)}   # the round in which a stage was armed last
            assert waited == last
    tc, la = _csrc("still_tc.cu"), _csrc("still_la_tc.cu")
    assert "mbar_drain_ring(bar.kv_full, kStages, armed, t0);" in tc.split("producer_role(", 1)[1].split("mma_role(", 1)[0]
    assert "mbar_drain_ring(full, 2, it, clock64());" in tc.split("score_select_tc_kernel(", 1)[1]
    scan = la.split("la_fused_kernel(", 1)[1]
    assert re.search(r"mbar_drain_ring\(x_full, 1, nx, t1\);\s*mbar_drain_ring\(u_full, n_stages, nu, t1\);", scan)


def test_tensor_map_rows_stay_below_the_guard():
    # Calls are taken up to B H N < 2^31 rows of a tensor, and a TMA row is a signed 32-bit coordinate.  So no map of the scan
    # spans more than one tensor of that many rows, and the row of its stores counts rows of one part.
    la = _csrc("still_la_tc.cu")
    assert "if ((long long)p->B * p->H * N >= (1ll << 31)) return STILL_ERR_UNSUPPORTED;" in la
    rows = re.findall(r"make_map_2d\(&t\w+, [^,]*(?:\([^)]*\))?[^,]*, ([^,]*),", la.split("int launch_fused(", 1)[1])
    assert len(rows) >= 8 and set(rows) <= {"BH * N", "BHkv * N", "(unsigned long long)p->H * D", "BH * (unsigned long long)sel_rows"}
    assert re.search(r"tma_store_2d\([^;]*, bh \* N \+ base\);", la)


def test_shared_arrays_that_vectors_are_stored_to_are_aligned():
    # A shared array is only as aligned as its element type unless it says more: those without an explicit alignment are
    # the ones that are accessed element by element (or, smem_raw, aligned by hand).
    plain = set()
    for name in os.listdir(still_build.CSRC):
        for m in re.finditer(r"__shared__ ([^;]*);", open(os.path.join(still_build.CSRC, name)).read()):
            if "__align__" not in m.group(1):
                plain.add(re.findall(r"(\w+)(?:\[[^\]]*\])*$", m.group(1))[0])
    assert plain == {"part", "smem_raw", "bar", "abort_word"}


def test_parameters_stay_a_plain_dataclass(lib):
    # A call leaves nothing among the fields, c() hands out a struct of the caller's own, and every call sees the fields as
    # they are, however they were set.
    import copy
    import dataclasses
    import pickle

    p = still.StillParams(2, 8, 2, 64, 64, 16, sm_scale=0.5)
    n = still.workspace_bytes(p, 1000)
    assert set(vars(p)) == {f.name for f in dataclasses.fields(p)}
    assert still.StillParams(**vars(p)) == p and dataclasses.replace(p, topk=8).topk == 8
    for q in (copy.copy(p), copy.deepcopy(p), pickle.loads(pickle.dumps(p))):
        assert q == p and still.workspace_bytes(q, 1000) == n
        q.B = 4
        assert still.workspace_bytes(q, 1000) > n and still.workspace_bytes(p, 1000) == n
    p.c().B = 0
    assert still.workspace_bytes(p, 1000) == n and p.c().B == 2
    vars(p)["B"] = 4
    assert still.workspace_bytes(p, 1000) > n
    p.sm_scale = 0.0
    assert still.workspace_bytes(p, 1000) == 0
    p.sm_scale = torch.tensor(0.0)          # a value that can change in place
    assert still.workspace_bytes(p, 1000) == 0
    p.sm_scale.fill_(0.5)
    assert still.workspace_bytes(p, 1000) > n
