"""What bench.py says about a profiled pass, on made-up launch counts: every variant of a call site goes to the kernel that ran
it, and the variants' bytes add up to the call site's.  And what it times: passes that have nothing left to set up."""
import numpy as np
import pytest

from paper_2503_05931_b200 import workloads as wl


def _profile(w, planes=128, heads=16):
    """Launch counts of a greedy pass of the bf16 library over the workload's row counts."""
    NL, out = w.model["n_layers"], {}
    add = lambda fam, n: out.setdefault(fam, {"ms": 1.0, "launches": 0}).__setitem__("launches", out.get(fam, {"launches": 0})["launches"] + n)
    for s in range(int(w.dec_lens.max())):
        rows = int((w.dec_lens > s).sum())
        v = "@plane" if rows > planes else "" if rows > 64 else "@gemv_staged" if rows > 4 else "@gemv"
        for site in ["qkv", "o", "oc", "ff1", "ff2"] + (["qc"] if rows > planes else []):
            add("gemm_" + site + v, NL)
        if rows > planes:
            add("layernorm@gamma", 3 * NL)
        add("attn_self" + ("@warp" if rows * heads > 1024 else ""), NL)
        add("attn_cross", NL)
        add("gemm_vocab" if rows > 16 else "gemm_vocab@gemv", 1)
        if rows > 16:
            add("layernorm", 1)
    add("precompute_cross_kv", 1)
    return out


@pytest.mark.parametrize("name", ["cfg2", "cfg3", "cfg4"])
def test_variants_share_a_call_sites_bytes(name):
    import bench
    w = wl.make_workload(name, with_weights=False, with_enc=False)
    prof = _profile(w)
    moved = bench.profile_bytes(prof, w)
    assert set(moved) == set(prof)
    for base in {f.partition("@")[0] for f in prof} - {"layernorm"}:
        total = sum(v for f, v in moved.items() if f.partition("@")[0] == base)
        want = bench.family_bytes(base, w)
        if base in ("gemm_qkv", "gemm_qc"):           # the query matrix is read by one of the two
            continue
        assert total == want, base
    both = sum(v for f, v in moved.items() if f.startswith(("gemm_qkv", "gemm_qc")))
    assert both == bench.family_bytes("gemm_qkv", w) + bench.family_bytes("gemm_qc", w)
    # many rows first: the early steps' short caches belong to the warp kernel
    if "attn_self@warp" in prof and "attn_self" in prof:
        n = prof["attn_self@warp"]["launches"] // w.model["n_layers"]
        assert moved["attn_self@warp"] == bench.family_bytes("attn_self", w, 0, n)


def test_kernel_names_exist_in_the_source():
    import glob
    import os
    import bench
    src = "".join(open(f).read() for f in glob.glob(os.path.join(os.path.dirname(bench.__file__), "paper_2503_05931_b200", "csrc", "*.cu*")))
    names = set(bench.KERNEL_OF_FAMILY.values()) | set(bench.KERNEL_OF_VARIANT.values()) | set(bench.NCU_TRAFFIC_RATIO) | {"vocab_gemv_kernel"}
    for name in names - {"step_rows/finish_step"}:
        assert name + "(" in src, name
    for variant in bench.KERNEL_OF_VARIANT:
        assert f'"@{variant}"' in src, variant
    assert set(bench.VARIANT_ORDER) | {"gamma"} == set(bench.KERNEL_OF_VARIANT) | {""}


@pytest.mark.parametrize("warmup, steps", [(3, 5), (4, 1)])
def test_timed_passes_do_not_set_anything_up(warmup, steps):
    """A pass from the host copies its inputs into a new device buffer while the decoder still holds the last one's: on a made-up
    clock the first two passes take a block of memory (60 ms each), later ones reuse it, and no timed pass may show it."""
    import bench
    clock, free, held, log = [0.0], [], [None], []

    class Event:
        def record(self):
            self.at = clock[0]

        def elapsed_time(self, other):
            return other.at - self.at

    def one_pass():
        if free:
            block = free.pop()
        else:
            block = object()
            clock[0] += 60.0
        if held[0] is not None:
            free.append(held[0])
        held[0] = block
        clock[0] += 10.0
        log.append("pass")

    total, per = bench.timed_passes(one_pass, warmup, steps, lambda: log.append("barrier"), Event, lambda: log.append("start"))
    assert log == ["pass"] * warmup + ["start", "barrier"] + ["pass"] * steps + ["barrier"]
    assert per == [10.0] * steps and total == 10.0 * steps
