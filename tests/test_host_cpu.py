"""The engine's host code without a GPU: its objects linked against a stand-in
for the CUDA runtime (``_fake_cudart.c``) in which kernels only leave their names
and an allocation can be made to fail."""
import ctypes
import glob
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))

INT8, BITPACK = 0, 1


@pytest.fixture(scope="module")
def fake_library(tmp_path_factory):
    from paper_cs_0312006_gb300 import _build
    objects = os.path.join(_build.OUT_DIR, "obj", "*.o")
    _build.build(force=len(glob.glob(objects)) != len(_build.sources()))
    out = str(tmp_path_factory.mktemp("host") / "libising_host.so")
    # -Bsymbolic: a CUDA runtime loaded earlier in the process does not take over
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-o", out,
                    os.path.join(HERE, "_fake_cudart.c"), *sorted(glob.glob(objects)),
                    "-lstdc++", "-lpthread", "-lm"], check=True)
    return out


@pytest.fixture()
def eng(fake_library, monkeypatch):
    from paper_cs_0312006_gb300 import _build, engine
    monkeypatch.setattr(_build, "LIB_PATH", fake_library)
    monkeypatch.setattr(engine, "_lib", None)
    lib = engine.load_library()
    lib.fake_launches.argtypes = [ctypes.c_char_p]
    lib.fake_fail_allocation(-1)
    lib.fake_clear_launches()
    yield engine
    lib.fake_fail_allocation(-1)
    lib.ising_clear_int8_configs()


def launches(eng, part):
    return eng.load_library().fake_launches(part.encode())


@pytest.mark.parametrize("cluster_size", [0, 2])
def test_failed_update_refuses_to_launch(eng, cluster_size):
    """Whichever allocation of an update fails, the batch launches nothing until
    an update succeeds; then it launches all of its lattices again."""
    lib = eng.load_library()
    few = [eng.Lattice(2, 64, 0.4, 1, layout=BITPACK)]
    many = [eng.Lattice(2, L, 0.4, L, layout=layout) for L in (32, 64, 130)
            for layout in (INT8, BITPACK)]
    failures = 0
    for k in range(20):
        batch = eng.Batch(few, 3, cluster_size=cluster_size, big_sites=1)
        batch.launch()
        lib.fake_fail_allocation(k)
        try:
            batch.update(many, 2)
        except eng.IsingError as e:
            failures += 1
            assert e.code == eng.ENOMEM
            assert not lib.fake_fail_pending()
            lib.fake_clear_launches()
            with pytest.raises(eng.IsingError) as refused:
                batch.launch()
            assert refused.value.code == eng.EINVAL
            assert launches(eng, "") == 0
            batch.sync()
            batch.update(many, 2)
        lib.fake_fail_allocation(-1)
        lib.fake_clear_launches()
        batch.launch()
        assert launches(eng, "joint_pass_kernel") == (4 if cluster_size == 0 else 0)
        batch.sync()
        batch.close()
    assert failures == (10 if cluster_size == 0 else 4)


def kernels_of(eng, lat, n):
    eng.load_library().fake_clear_launches()
    lat.sweep(n, 1)
    return {part: launches(eng, part) for part in ("resident_kernel", "pass_int8_strip",
                                                   "pass_int8_vecs", "pass_int8_tma",
                                                   "pass_packed")
            if launches(eng, part)}


@pytest.mark.parametrize("dims,L", [(2, 64), (2, 160), (2, 512), (3, 32), (3, 64)])
def test_chosen_kernel_runs(eng, dims, L):
    """Runs of sweeps of small lattices are one launch, unless the caller names an
    int8 kernel or registers a configuration: then its passes run."""
    strip, staged, whole = {"pass_int8_strip": 8}, {"pass_int8_tma": 8}, {"resident_kernel": 1}
    assert kernels_of(eng, eng.Lattice(dims, L, 0.3, 1), 4) == whole
    for kernel, want in ((eng.KERNEL_STRIP, strip), (eng.KERNEL_TMA, staged)):
        lat = eng.Lattice(dims, L, 0.3, 1, kernel=kernel)
        assert kernels_of(eng, lat, 4) == want
        lat.set_kernel(eng.KERNEL_AUTO)
        assert kernels_of(eng, lat, 4) == whole
    lat = eng.Lattice(dims, L, 0.3, 1)
    packed = eng.Lattice(dims, L, 0.3, 1, layout=BITPACK)
    as_before = kernels_of(eng, packed, 4)
    eng.set_int8_config(dims, L, L, eng.KERNEL_TMA, tile_rows=1)
    assert kernels_of(eng, lat, 4) == staged
    assert kernels_of(eng, packed, 4) == as_before  # the choice is about int8 passes
    eng.set_int8_config(dims, L, L, eng.KERNEL_STRIP)
    assert kernels_of(eng, lat, 4) == strip
    eng.clear_int8_configs()
    assert kernels_of(eng, lat, 4) == whole


def batch_launches(eng, specs, **opts):
    """Launches of a batch of (dims, L, sweeps, copies[, rule]): joint passes, the
    persistent kernel, and the lattices counted as large and as small."""
    lats, sweeps = [], []
    for dims, L, n, copies, *rule in specs:
        for k in range(copies):
            lats.append(eng.Lattice(dims, L, 0.3, k, layout=BITPACK, rule=rule[0] if rule else 0))
            sweeps.append(n)
    batch = eng.Batch(lats, sweeps, use_graph=False, **opts)
    eng.load_library().fake_clear_launches()
    batch.launch()
    info = batch.info()
    batch.close()
    return (launches(eng, "joint_pass_kernel"), launches(eng, "batch_kernel"), info["n_big"],
            info["n_small"])


def test_batch_routes(eng):
    """Which lattices of a batch take joint passes when the caller names no cluster
    size: those that would keep a queue of CTAs waiting, not small ones beside
    them that run longer, and none where the queue fills the GPU or waits for a
    small one all the same."""
    assert batch_launches(eng, [(2, 64, 5000, 4)]) == (0, 1, 0, 4)
    assert batch_launches(eng, [(2, 512, 30, 16)]) == (60, 0, 16, 0)
    assert batch_launches(eng, [(2, 1024, 100, 4), (2, 64, 300, 4)]) == (200, 1, 4, 4)
    assert batch_launches(eng, [(2, 512, 30, 16), (2, 64, 5000, 4)]) == (0, 1, 16, 4)
    assert batch_launches(eng, [(2, 256, 10, 1024)]) == (0, 1, 0, 1024)
    assert batch_launches(eng, [(2, 1024, 10, 256)]) == (0, 1, 256, 0)  # clusters of four
    # each update rule for itself
    assert batch_launches(eng, [(2, 512, 30, 16), (2, 64, 500, 4, 1)]) == (60, 1, 16, 4)
    # a size to go by, or a cluster size
    assert batch_launches(eng, [(2, 64, 5, 4)], big_sites=1) == (10, 0, 4, 0)
    assert batch_launches(eng, [(2, 64, 5, 4), (2, 32, 7, 3)], big_sites=4096) == (10, 1, 4, 3)
    assert batch_launches(eng, [(2, 512, 30, 16)], cluster_size=2) == (0, 1, 16, 0)
    assert batch_launches(eng, [(2, 512, 0, 16)])[0] == 0


def test_tuner_can_choose_the_default(monkeypatch):
    """A batch run with no options is among what the batch tuner compares."""
    from paper_cs_0312006_gb300 import autotune, workloads

    def run_batched(specs, opts, launches, layout):
        return (1.0 if opts.get("cluster_size") or opts.get("big_sites") else 0.5), []

    monkeypatch.setattr(autotune.batched, "run_batched", run_batched)
    monkeypatch.setattr(autotune, "_device_name", lambda: "none")
    best = autotune.tune(workloads.batched_mix(8, 10), use_cache=False)["opts"]
    assert not best["cluster_size"] and not best["big_sites"] and not best["block_threads"]
