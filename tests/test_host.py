"""CPU-side checks: the C-ABI library loads and exports what the header declares, the binding
refuses to run without CUDA, the input generator is deterministic, and the sequence sharding
used for more than one GPU reproduces the single-process result (gloo, world_size 2)."""
import ctypes
import os
import re
import subprocess
import sys
import sysconfig

import numpy as np
import pytest
import torch

import gen

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared_symbols():
    text = open(os.path.join(ROOT, "include", "picospec.h")).read()
    return sorted(set(re.findall(r"PICOSPEC_API\s+[\w\s\*]+?\b(picospec_\w+)\s*\(", text)))


def test_library_exports_every_declared_symbol():
    from paper_2603_19133_b200 import buildlib
    lib = ctypes.CDLL(buildlib.build())
    names = _declared_symbols()
    assert {"picospec_compress", "picospec_verify", "picospec_residual_sample", "picospec_create",
            "picospec_destroy", "picospec_status", "picospec_strerror"} <= set(names)
    for n in names:
        assert hasattr(lib, n), f"{n} declared in picospec.h but not exported"
    lib.picospec_strerror.restype = ctypes.c_char_p
    assert lib.picospec_strerror(0) == b"ok"
    assert b"capacity" in lib.picospec_strerror(-3)


def test_only_the_c_abi_is_exported():
    from paper_2603_19133_b200 import buildlib
    out = subprocess.run(["nm", "-D", "--defined-only", buildlib.build()], capture_output=True, text=True).stdout
    exported = [ln.split()[-1] for ln in out.splitlines() if " T " in ln]
    assert sorted(exported) == _declared_symbols()


def test_host_argument_checks_need_no_gpu():
    from paper_2603_19133_b200 import buildlib
    lib = ctypes.CDLL(buildlib.build())
    h = ctypes.c_void_p()
    assert lib.picospec_create(None, 0, 1, 1, 1000, 8) == -1
    assert lib.picospec_create(ctypes.byref(h), 0, 0, 1, 1000, 8) == -1          # max_batch <= 0
    assert lib.picospec_create(ctypes.byref(h), 0, 1, 1, 1000, 5000) == -1       # max_k too large
    assert lib.picospec_destroy(None) == -1


def test_a_marshaller_of_another_torch_is_not_loaded(monkeypatch):
    from paper_2603_19133_b200 import binding, buildlib
    binding.lib()
    here = buildlib.marshal_path()
    assert os.path.exists(here) and here.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    built = []
    with monkeypatch.context() as m:
        m.setattr(torch, "__version__", "0.0.1+other")
        m.setattr(binding, "_lib", None)
        m.setattr(binding, "_marshal", None)
        m.setattr(buildlib, "build", lambda *a, **k: built.append(buildlib.marshal_path()) or buildlib.LIB)
        assert buildlib.marshal_path() != here
        with pytest.raises(ImportError):        # (nothing was built for that version here)
            binding.lib()
        assert built == [buildlib.marshal_path()] and binding._lib is None
    binding.lib()


@pytest.mark.skipif(torch.cuda.is_available(), reason="checks the behaviour without a GPU")
def test_no_cpu_fallback():
    import paper_2603_19133_b200 as ps
    with pytest.raises(RuntimeError):
        ps.Context(1, 1, 1000, 8)


def test_product_package_never_touches_the_oracle():
    pkg = os.path.join(ROOT, "paper_2603_19133_b200")
    for dirpath, _, files in os.walk(pkg):
        for f in files:
            if f.endswith((".py", ".cu", ".cuh", ".h")):
                text = open(os.path.join(dirpath, f)).read()
                assert "oracle" not in text.lower(), f"{f} mentions the oracle"


def test_generator_is_deterministic_and_shaped():
    w = gen.scaled(gen.WORKLOADS["config2"], B=2, V=5000)
    a, b = gen.make_inputs(w, 5), gen.make_inputs(w, 5)
    c = gen.make_inputs(w, 6)
    for k in a:
        assert torch.equal(a[k], b[k])
    assert not torch.equal(a["draft_logits"], c["draft_logits"])
    assert a["draft_logits"].shape == (2, w.G, 5000) and a["draft_logits"].dtype == torch.bfloat16
    assert a["target_logits"].shape == (2, w.G + 1, 5000)
    for k in ("u_draft", "u_accept", "u_resample"):
        assert a[k].dtype == torch.float32 and float(a[k].min()) >= 0 and float(a[k].max()) < 1
    # long tail: the largest logit stands well above the median
    l = a["draft_logits"].float()
    assert float((l.max(-1).values - l.median(-1).values).min()) > 5
    w4 = gen.scaled(gen.WORKLOADS["config4"], B=3, V=3000)
    d = gen.make_inputs(w4, 1)
    T = d["temperature"].numpy()
    assert np.all((T >= 0.5) & (T <= 1.2)) and len(set(T.tolist())) == 3


def test_shard_ranges_partition_the_batch():
    from paper_2603_19133_b200.shard import shard_range
    for B in (0, 1, 7, 8, 256, 511):
        for world in (1, 2, 3, 8):
            ranges = [shard_range(B, r, world) for r in range(world)]
            assert ranges[0][0] == 0 and ranges[-1][1] == B
            assert all(a[1] == b[0] for a, b in zip(ranges, ranges[1:]))
            sizes = [b1 - b0 for b0, b1 in ranges]
            assert max(sizes) - min(sizes) <= 1


_WORKER = r'''
import os, sys
sys.path.insert(0, sys.argv[1])
import numpy as np, torch, torch.distributed as dist
import gen, oracle
from paper_2603_19133_b200.shard import shard_range, gather_sequences, max_over_ranks
dist.init_process_group("gloo")
rank, world = dist.get_rank(), dist.get_world_size()
w = gen.Workload("t", V=3000, B=7, G=3, dtype="bf16", s=1.1, sigma_d=1.5, corr=0.8, sigma_t=1.0, T=None,
                 top_k=0, top_p=0.9, k_max=16)
inp = gen.make_inputs(w, 11)                       # every rank generates the same global batch
f = lambda t: t.float().numpy() if t.is_floating_point() else t.numpy()
b0, b1 = shard_range(w.B, rank, world)
loc = {k: f(v[b0:b1]) for k, v in inp.items()}
# the CPU stand-in for the per-rank GPU call: each rank works on its own block of sequences only
qi, qp, qc, tok = oracle.compress(loc["draft_logits"], loc["temperature"], w.top_k, w.top_p, w.k_max, loc["u_draft"])
r = oracle.verify(loc["target_logits"], loc["temperature"], tok, qi, qp, qc, loc["u_accept"], loc["u_resample"])
alen = gather_sequences(torch.from_numpy(r["accept_len"]), w.B)
token = gather_sequences(torch.from_numpy(r["token"]), w.B)
pd = gather_sequences(torch.from_numpy(r["p_draft"]), w.B)
t = max_over_ranks(1.0 + rank)
if rank == 0:
    full = {k: f(v) for k, v in inp.items()}
    qi, qp, qc, tok = oracle.compress(full["draft_logits"], full["temperature"], w.top_k, w.top_p, w.k_max, full["u_draft"])
    ref = oracle.verify(full["target_logits"], full["temperature"], tok, qi, qp, qc, full["u_accept"], full["u_resample"])
    assert np.array_equal(alen.numpy(), ref["accept_len"]) and np.array_equal(token.numpy(), ref["token"])
    assert np.array_equal(pd.numpy(), ref["p_draft"])
    assert t == float(world)
    print("SHARD_OK")
dist.destroy_process_group()
'''


def test_sequence_sharding_world_size_2_gloo(tmp_path):
    script = tmp_path / "worker.py"
    script.write_text(_WORKER)
    cmd = [sys.executable, "-m", "torch.distributed.run", "--nnodes=1", "--nproc-per-node=2",
           "--master-addr", "127.0.0.1", "--master-port", "29571", str(script), ROOT]
    run = subprocess.run(cmd, capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stdout[-2000:] + run.stderr[-2000:]
    assert "SHARD_OK" in run.stdout


_VP_WORKER = r'''
import os, sys
sys.path.insert(0, sys.argv[1])
import numpy as np, torch, torch.distributed as dist
import gen, oracle
from oracle import vocab_parallel as ovp
from paper_2603_19133_b200 import vocab_parallel as vp
dist.init_process_group("gloo")
rank, world = dist.get_rank(), dist.get_world_size()
w = gen.Workload("t", V=5120 + 300, B=5, G=3, dtype="f32", s=1.1, sigma_d=1.5, corr=0.8, sigma_t=1.0, T=None,
                 top_k=0, top_p=0.9, k_max=24)
inp = gen.make_inputs(w, 21)                       # every rank generates the same global batch ...
f = lambda t: t.float().numpy() if t.is_floating_point() else t.numpy()
T = f(inp["temperature"])
qi, qp, qc, tok = oracle.compress(f(inp["draft_logits"]), T, w.top_k, w.top_p, w.k_max, f(inp["u_draft"]))
v0, v1 = vp.slice_bounds(w.V, world, rank)         # ... and keeps its own slice of the target logits only
sl = np.ascontiguousarray(f(inp["target_logits"])[:, :, v0:v1])
cpr = vp.chunks_per_rank(w.V, world)
exch = vp.DistExchange()
# the CPU stand-in for the per-rank kernels, the product's exchanges between them
m, s = ovp.slice_records(sl, T)
pad = cpr - m.shape[-1]
rec = np.stack([np.pad(m, ((0, 0), (0, 0), (0, pad)), constant_values=-np.inf), np.pad(s, ((0, 0), (0, 0), (0, pad)))], -1)
(rec_all,) = exch.gather([torch.from_numpy(rec)])                       # [world, B, G+1, cpr, 2]
(ent_all,) = exch.maximum([torch.from_numpy(ovp.slice_entries(sl, v0, tok, qi, qc))])
nch = (w.V + 1023) // 1024
ra = rec_all.numpy()
m_all = np.concatenate([ra[r, ..., 0] for r in range(world)], -1)[..., :nch]
s_all = np.concatenate([ra[r, ..., 1] for r in range(world)], -1)[..., :nch]
owner = np.arange(nch) // cpr
d = ovp.decide(m_all, s_all, ent_all.numpy(), T, tok, qi, qp, qc, f(inp["u_accept"]), f(inp["u_resample"]), owner)
mine = ovp.draw_in_slice(sl, v0, rank, d, T, qi, qp, qc, f(inp["u_resample"]))
(token,) = exch.maximum([torch.from_numpy(mine)])
ref = oracle.verify(f(inp["target_logits"]), T, tok, qi, qp, qc, f(inp["u_accept"]), f(inp["u_resample"]))
assert np.array_equal(d["accept_len"], ref["accept_len"]) and np.array_equal(token.numpy(), ref["token"])
assert (mine >= 0).sum() < w.B or world == 1      # no rank owns every picked chunk
np.testing.assert_allclose(d["p_draft"], ref["p_draft"], rtol=1e-12)
if rank == 0:
    print("VP_OK")
dist.destroy_process_group()
'''


def test_vocabulary_parallel_exchange_world_size_2_gloo(tmp_path):
    # the product's exchange code (all-gather of chunk records, element-wise maximum of gathered logits and
    # of tokens) between two gloo ranks on CPU tensors, with the oracle's per-slice routines standing in for
    # the kernels: the result equals plain verification of the whole vocabulary
    script = tmp_path / "vp_worker.py"
    script.write_text(_VP_WORKER)
    cmd = [sys.executable, "-m", "torch.distributed.run", "--nnodes=1", "--nproc-per-node=2",
           "--master-addr", "127.0.0.1", "--master-port", "29573", str(script), ROOT]
    run = subprocess.run(cmd, capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stdout[-2000:] + run.stderr[-2000:]
    assert "VP_OK" in run.stdout


def test_bench_starts_its_own_ranks_for_more_than_one_gpu():
    # `bench.py --gpus 2` without a torchrun environment starts two ranks of itself; the reference arm
    # needs no GPU (rank 0 alone times the oracle, the other rank leaves without work), so the launcher
    # path runs here as it is
    import json
    env = {k: v for k, v in os.environ.items() if k not in ("RANK", "LOCAL_RANK", "WORLD_SIZE")}
    cmd = [sys.executable, os.path.join(ROOT, "bench.py"), "--gpus", "2", "--impl", "reference", "--steps", "1",
           "--warmup", "0", "--workload", "config1", "--ref-sample", "1"]
    run = subprocess.run(cmd, capture_output=True, text=True, timeout=600, env=env)
    assert run.returncode == 0, run.stdout[-2000:] + run.stderr[-2000:]
    lines = [ln for ln in run.stdout.splitlines() if ln.startswith("{")]
    assert len(lines) == 1                      # one JSON line, from rank 0
    line = json.loads(lines[0])
    assert line["impl"] == "reference" and line["n_gpus"] == 2 and line["ranks_launched"] == 2
    assert line["config"]["parallelism"].startswith("dp2")


def test_bench_reads_ncu_traffic_only_for_unchanged_kernels(tmp_path, monkeypatch):
    sys.path.insert(0, ROOT)
    import bench
    h = bench.source_hash(["verify_kernels.cuh"])
    prof = tmp_path / "profiles"
    prof.mkdir()
    (prof / "a.md").write_text(f"x\nbench-traffic: kernel=k1 workload=config4 bytes=123 sources=verify_kernels.cuh hash={h}\n"
                               "bench-traffic: kernel=k2 workload=config4 bytes=5 sources=verify_kernels.cuh hash=000000000000\n")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.ncu_traffic("config4", "k1") == 123
    assert bench.ncu_traffic("config4", "k2") is None        # the kernel changed since the capture
    assert bench.ncu_traffic("config3", "k1") is None


def test_throughput_calculator_matches_the_term_by_term_oracle():
    # the product's closed forms (Sec. 3.4, Eqs. 5-10) against the oracle's sums and case analysis
    from paper_2603_19133_b200 import perf_model as pm
    from oracle import wire
    import itertools
    for alpha, gamma in itertools.product((0.0, 0.2, 0.7, 0.95, 1.0), (1, 4, 6, 9)):
        assert abs(pm.expected_length(alpha, gamma) - wire.expected_length(alpha, gamma)) < 1e-9
        for td, tr, tv in ((40.0, 25.0, 10.0), (5.0, 50.0, 8.0), (30.0, 0.0, 30.0)):
            assert abs(pm.throughput_sync(alpha, gamma, td, tr, tv) - wire.throughput_sync(alpha, gamma, td, tr, tv)) < 1e-12
            assert abs(pm.expected_time_async(alpha, gamma, td, tr, tv) - wire.expected_time_async(alpha, gamma, td, tr, tv)) < 1e-9
            assert abs(pm.speedup(alpha, gamma, td, tr, tv) - wire.speedup(alpha, gamma, td, tr, tv)) < 1e-9
    assert abs(pm.speedup(1.0, 5, 40.0, 25.0, 10.0) - pm.speedup_limit(40.0, 25.0, 10.0)) < 1e-12
    # payload sizes: the wire message of K = 10 pairs, against the oracle's packer and the C helper
    import numpy as np
    qi = np.arange(10, dtype=np.int32).reshape(1, 10)
    qp = np.full((1, 10), 0.1, np.float32)
    for fp16 in (False, True):
        assert pm.downlink_bytes(10, fp16) == wire.pack(qi, qp, np.array([10]), int(fp16)).size
    from paper_2603_19133_b200 import buildlib
    lib = ctypes.CDLL(buildlib.build())
    lib.picospec_wire_bytes.restype = ctypes.c_longlong
    lib.picospec_wire_bytes.argtypes = [ctypes.c_int, ctypes.c_longlong, ctypes.c_int]
    for rows, n, pt in ((1, 10, 0), (1, 10, 1), (7, 33, 1), (1536, 1536 * 256, 0), (0, 0, 0)):
        assert lib.picospec_wire_bytes(rows, n, pt) == wire.wire_size(rows, n, pt)
    assert lib.picospec_wire_bytes(-1, 0, 0) == -1 and lib.picospec_wire_bytes(1, 1, 2) == -1
    assert pm.dense_row_bytes(128256) / pm.downlink_bytes(10, True) > 1000
