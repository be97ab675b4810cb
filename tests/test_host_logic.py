"""Host-side checks that need no GPU: the CUDA library loads, exports every symbol the header declares,
rejects bad configurations before touching a device, and sizes its workspace sensibly."""
import ctypes as C
import os
import re

import pytest

from paper_2503_01840_b200 import binding as sb
from paper_2503_01840_b200 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_library_exports_every_declared_symbol():
    hdr = open(os.path.join(ROOT, "include", "spec_b200.h")).read()
    declared = set(re.findall(r"\b(spec_[a-z_0-9]+)\s*\(", hdr))
    declared -= {"spec_ctx"}
    L = sb.lib()
    assert declared, "no declarations found"
    for name in sorted(declared):
        assert hasattr(L, name), f"{name} is declared in spec_b200.h but not exported"
    assert set(sb.EXPORTS) == declared


def test_workspace_bytes_and_cfg_validation():
    L = sb.lib()
    cfg = sb.make_cfg(synth.C1, batch=1, max_ctx=256, num_pages=16)
    n = L.spec_workspace_bytes(C.byref(cfg))
    assert n > 0 and n % 256 == 0
    cfg2 = sb.make_cfg(synth.C1, batch=1, max_ctx=256, num_pages=32)
    kv_page = synth.C1.n_kv_heads * synth.C1.page_size * synth.C1.head_dim * 4
    grow = L.spec_workspace_bytes(C.byref(cfg2)) - n
    assert grow == 16 * kv_page * 2 * (synth.C1.n_layers + 1)     # K and V pools of every layer + the draft layer
    for field, bad in (("tree_nodes", 65), ("tree_topk", 0), ("tree_depth", 0), ("head_dim", 60), ("page_size", 24),
                       ("dtype", 7), ("n_kv_heads", 3), ("batch", 0)):
        c = sb.make_cfg(synth.C1, batch=1, max_ctx=256, num_pages=16)
        setattr(c, field, bad)
        assert L.spec_workspace_bytes(C.byref(c)) == 0, field


def test_init_rejects_bad_arguments_without_a_device():
    L = sb.lib()
    h = C.c_void_p()
    assert L.spec_init(C.byref(h), None, None, None) == -2
    cfg = sb.make_cfg(synth.C1, batch=1, max_ctx=256, num_pages=16)
    tw, dw = sb._TW(), sb._DW()
    cfg.tree_nodes = 100
    assert L.spec_init(C.byref(h), C.byref(tw), C.byref(dw), C.byref(cfg)) == -1
    assert b"tree_nodes" in L.spec_last_error(None)
    cfg.tree_nodes = 16
    assert L.spec_init(C.byref(h), C.byref(tw), C.byref(dw), C.byref(cfg)) == -2      # workspace NULL
    cfg.workspace, cfg.workspace_bytes = 4096 + 8, 1 << 20
    assert L.spec_init(C.byref(h), C.byref(tw), C.byref(dw), C.byref(cfg)) == -3      # misaligned
    cfg.workspace = 4096
    assert L.spec_init(C.byref(h), C.byref(tw), C.byref(dw), C.byref(cfg)) == -2      # NULL weights
    assert not h.value


def test_paper_shaped_workspaces_fit_one_gpu():
    L = sb.lib()
    for name, reserve in (("C2", 256), ("C3", 128), ("C4", 1024), ("C5", 128)):
        m = synth.CONFIGS[name]
        plen = m.prompt_hi if m.batch > 1 else m.prompt_len
        max_ctx = plen + reserve + 160
        pages = m.batch * ((max_ctx + m.page_size - 1) // m.page_size)
        cfg = sb.make_cfg(m, batch=m.batch, max_ctx=max_ctx, num_pages=pages)
        n = L.spec_workspace_bytes(C.byref(cfg))
        assert 0 < n < 40e9, (name, n)


def test_single_kernel_entry_points_reject_null():
    L = sb.lib()
    assert L.spec_gemm(1, 0, None, None, None, 1, 1, 8, 1, None, None) == -2
    assert L.spec_argmax(None, 1, 1, None, None) == -2
    assert L.spec_logsoftmax_topk(None, 1, 1, 1, None, None, None, None) == -2
    assert L.spec_gemm_fused(None, None, None, 1, 1, 8, 1, 0, 0, None) == -2
    assert L.spec_gemm_swiglu(None, None, None, None, 1, 128, 8, None) == -2
    assert L.spec_step_sampled(None, 1.0, None, None, None) == -2
    assert L.spec_topk_scratch_bytes(10, 32000, 10) > 0


def _kernel_bodies():
    """(file, kernel name, body text) of every __global__ function of the CUDA sources."""
    csrc = os.path.join(ROOT, "paper_2503_01840_b200", "csrc")
    for fn in sorted(os.listdir(csrc)):
        if not fn.endswith(".cu"):
            continue
        s = open(os.path.join(csrc, fn)).read()
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(", s):
            i = s.index("{", m.end())
            depth, j = 0, i
            while True:
                depth += {"{": 1, "}": -1}.get(s[j], 0)
                if depth == 0:
                    break
                j += 1
            yield fn, m.group(1), s[i:j]


def test_every_step_kernel_orders_itself_behind_its_predecessor():
    """Kernels of a step are launched with programmatic dependent launch: a kernel may start before its predecessor
    has finished, and its successor waits only for IT.  A kernel without griddepcontrol.wait would let its successor
    overtake the kernel before it (the first QKV GEMM reading a RoPE table that is still being written), so every
    kernel the scheduler launches with the attribute must wait, and must do so before it touches what a kernel of the step
    wrote.  The GEMMs read weights before it, the attention kernels what the next test names."""
    never_pdl = {"gemm_tcgen05_kernel", "reduce_slices_kernel"}      # launched without the attribute
    seen = 0
    for fn, name, body in _kernel_bodies():
        if name in never_pdl:
            continue
        seen += 1
        assert "pdl_wait()" in body, f"{fn}: {name} never calls pdl_wait()"
        assert "pdl_trigger()" in body, f"{fn}: {name} never calls pdl_trigger()"
    assert seen >= 25
    # the elementwise / tree kernels wait first thing: nothing but declarations may precede the wait
    for fn, name, body in _kernel_bodies():
        if fn in ("elementwise.cu", "tree.cu", "gemm_ref.cu", "attn_ref.cu") and name not in never_pdl:
            head = body[: body.index("pdl_wait()")]
            head = "\n".join(l for l in head.split("\n") if "__shared__" not in l)
            assert "[" not in head and "->" not in head, f"{fn}: {name} touches memory before pdl_wait()"


def test_attention_reads_ahead_only_behind_launches_that_wait_first():
    """The attention kernels of attn_fast.cu read row metadata, the page table and cached context before their wait.  That holds only
    while the launch in front lets its dependents start after its own wait (everything before it is complete then), and while
    nothing that launch writes is read early."""
    bodies = {name: body for _, name, body in _kernel_bodies()}
    early = [n for n in ("attn_tma_kernel", "attn_umma_kernel", "attn_tma_small_kernel") if "p.m.seq" in bodies[n][: bodies[n].index("pdl_wait()")]]
    assert len(early) == 3, early
    for name in early:
        head = bodies[name][: bodies[name].index("pdl_wait()")]
        for written_in_front in ("p.q ", "p.q+", "p.out", "part_o", "part_ml"):
            assert written_in_front not in head, f"{name} touches {written_in_front} before its wait"
        assert "p.ctx_ready ? ctx : 0" in head and "ctx_early" in bodies[name], name
    # the launches in front of an attention launch
    for name, epi in (("gemm_fused_kernel", "EPI_QKV"), ("gemm_wide_kernel", "WIDE_QKV"), ("gemm_wide_split_kernel", "WIDE_QKV")):
        lines = [l.strip() for l in bodies[name].split("\n")]
        at = [i for i, l in enumerate(lines) if "pdl_trigger()" in l]
        for i in at:
            if lines[i].startswith(f"if (EPI != {epi}) pdl_trigger();"):
                continue
            assert lines[i].startswith(f"if (EPI == {epi}) pdl_trigger();") and lines[i - 1] == "pdl_wait();", f"{name}: {lines[i]}"
        assert len(at) >= 3, name
    body = bodies["rope_kv_kernel"]
    assert body.index("pdl_wait()") < body.index("pdl_trigger()")
    # and nothing is launched between the two
    api = open(os.path.join(ROOT, "paper_2503_01840_b200", "csrc", "api.cu")).read()
    calls = [m.start() for m in re.finditer(r"\n\s+attention\(pool, rows, tail_len\);", api)]
    assert len(calls) == 3
    for c in calls:
        before = [m for m in re.finditer(r"(\w+)(?:<T>)?\(", api[:c]) if m.group(1) in ("fgemm", "wgemm", "gemm", "gemm_cat") or m.group(1).startswith("launch_")]
        last = before[-1]
        assert last.group(1) in ("launch_rope_kv", "launch_norm_qkv") or api[last.end():].startswith("EPI_QKV"), last.group(1)


def test_scores_are_waited_for_in_the_straight_line_of_their_loads():
    """Before tcgen05.wait::ld nothing may read what a load puts out, not even a copy that the compiler puts where two paths with a load each come
    together.  So the causal kernel's loads are followed by their wait in the same straight line, and the scores are pinned behind it."""
    body = {name: body for _, name, body in _kernel_bodies()}["attn_causal_kernel"]
    loads = [m for m in re.finditer(r"tmem_ld32\([^;]*\);", body)]
    assert len(loads) >= 3
    for m in loads:
        between = body[m.end(): body.index("tmem_ld_wait();", m.end())]
        assert not re.sub(r"tmem_ld32\([^;]*\);", "", between).strip(), between
    assert re.search(r"tmem_ld_wait\(\);\s+pin32\(s\);\s+pin32\(s \+ 32\);", body)


def test_clock_record_of_a_short_timed_region(tmp_path, monkeypatch):
    """A region of 0.1 s has samples of its own, however long nvidia-smi takes to start (a stand-in for it here)."""
    import time
    fake = tmp_path / "nvidia-smi"
    fake.write_text('#!/bin/bash\nsleep 0.3\necho "0, 600, 1965, 200.0, 0x1, Not Active, Not Active, Not Active, Not Active"\n'
                    'while [ ! -e "%s" ]; do sleep 0.01; done\n'
                    'while true; do echo "0, 1900, 1965, 900.0, 0x4, Not Active, Not Active, Not Active, Active"; sleep 0.01; done\n' % (tmp_path / "busy"))
    fake.chmod(0o755)
    monkeypatch.setenv("PATH", f"{tmp_path}:{os.environ['PATH']}")
    monkeypatch.syspath_prepend(ROOT)
    import bench
    sampler = bench.ClockSampler(0)
    sampler.mark()
    (tmp_path / "busy").write_text("")
    time.sleep(0.3)
    out = sampler.stop()
    assert out["samples"] >= 2 and out["sm_mhz"] == 1900 and out["sm_max_mhz"] == 1965 and out["reasons"] == ["sw_power_cap"], out
