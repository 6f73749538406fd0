"""The checked build of the library (liblqer_dbg.so, -DLQER_DEBUG_BOUNDS): every global store of the inference
kernels and every copy of packed weights checks its byte range against the extent of its buffer; a violation goes to
the status word and the access is skipped.  It stands in for a memory checker.

The library is process wide, so the checked build runs in child processes (LQER_DEBUG_BOUNDS=1 makes the binding
load it): the small parity cases of the main suite must pass under it with a clean status word, and a launch whose Y is
declared shorter than it is (the build's own test hook) must report LQER_ERR_BOUNDS, leave the bytes beyond the
declared extent untouched and leave the context usable.
"""
import os
import subprocess
import sys
import textwrap

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _run(args, timeout=900):
    env = dict(os.environ, LQER_DEBUG_BOUNDS="1")
    return subprocess.run([sys.executable, *args], cwd=ROOT, env=env, capture_output=True, text=True, timeout=timeout)


def test_small_parity_cases_pass_under_the_checked_build():
    # every path of the layer on the small specs: prepare, both prologues, both GEMMs, the decode kernels, shared
    # launches, bf16 and MXINT8 boundaries; each test polls the status word, so a bounds report fails it
    r = _run(["-m", "pytest", "-x", "-q", "-m", "gpu",
              "tests/test_gpu_parity.py", "tests/test_gpu_bf16_io.py", "tests/test_gpu_mxint8_io.py", "tests/test_gpu_w2.py",
              "tests/test_gpu_small_mma.py", "tests/test_gpu_small_batches.py", "tests/test_gpu_digit_prologue.py",
              "tests/test_gpu_decode_cluster.py", "tests/test_gpu_pair_tiles.py", "tests/test_gpu_batched_mixed_rows.py",
              "tests/test_gpu_cluster_stages.py", "tests/test_gpu_small_sums.py",
              "-k", "not full and not stack and not sweep and not round"])
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]
    assert " passed" in r.stdout


def test_a_short_extent_is_reported_and_nothing_beyond_it_is_written():
    code = textwrap.dedent("""
        import numpy as np, torch
        import lqer_inputs as gen
        import paper_2402_02446_b200 as L
        from paper_2402_02446_b200 import binding
        assert binding.DEBUG_BOUNDS and L.lib_path().endswith("liblqer_dbg.so")
        E = binding.STATUS_NAMES.index
        dev = "cuda:0"
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
        for M, path in ((3, binding.PATH_AUTO), (3, binding.PATH_DECODE), (9, binding.PATH_SMALL), (40, binding.PATH_AUTO), (300, binding.PATH_AUTO)):
            spec = gen.LayerSpec("short", M=M, K=512, N=384, k=16, calib_rows=32, outlier_frac=0.01, outlier_scale=20.0, seed=501)
            W = gen.make_weight(spec); A, B = gen.make_random_factors(spec)
            Pg = L.prepare_weights(t(W), t(A), t(B))
            X = t(gen.make_activations(spec))
            ws = L.new_workspace(M, Pg)
            L.set_path(path)
            Y_good = L.linear(X, Pg, ws).clone()
            assert L.poll_status(ws) == 0
            cut = 4 * 100                                   # the last hundred floats of Y are declared out of range
            Y = torch.full((M, spec.N), 7.0, dtype=torch.float32, device=dev)
            L.debug_bounds_shrink(cut)
            try:
                L.linear(X, Pg, ws, Y)
                torch.cuda.synchronize()
            finally:
                L.debug_bounds_shrink(0)
            assert L.poll_status(ws) == E("LQER_ERR_BOUNDS"), (M, L.poll_status(ws))
            flat, good = Y.flatten(), Y_good.flatten()
            assert torch.all(flat[-100:] == 7.0)            # the guarded stores were skipped
            assert torch.equal(flat[:-128], good[:-128])    # everything clear of the cut was written as usual
            assert L.lib().lqer_workspace_init(ws.data_ptr(), ws.numel(), None) == 0
            assert torch.equal(L.linear(X, Pg, ws), Y_good) and L.poll_status(ws) == 0
            L.set_path(binding.PATH_AUTO)
            Pg.release()
        print("checked-build-ok")
    """)
    r = _run(["-c", code])
    assert r.returncode == 0 and "checked-build-ok" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]


def test_converter_warps_that_come_late_to_a_batch_lose_nothing():
    # three tiles per CTA, a tile being a batch of four slabs, one of one and one of two rank slabs: groups of converter
    # warps sit batches out in every ring (four, three and two slots).  They look at those batches some 50 us late, long
    # after the slot could have been filled again: the result must be the undelayed one, and no wait may run out.
    code = textwrap.dedent("""
        import torch
        import paper_2402_02446_b200 as L
        dev = "cuda:0"
        K, N, k = 320, 3 * 148 * 256, 72
        g = torch.Generator(device=dev); g.manual_seed(7)
        draw = lambda *s: torch.randn(s, generator=g, device=dev)
        Pg = L.prepare_weights(draw(K, N) * 0.02, draw(K, k) / K ** 0.5, draw(k, N) * 0.01)
        for M in (20, 64, 100):
            X = draw(M, K)
            ws = L.new_workspace(M, Pg)
            Y = L.linear(X, Pg, ws).clone()
            assert L.poll_status(ws) == 0
            L.debug_converter_lag(100_000)
            try:
                late = L.linear(X, Pg, ws)
                assert L.poll_status(ws) == 0, M
            finally:
                L.debug_converter_lag(0)
            assert torch.equal(late, Y), M
        print("late-converters-ok")
    """)
    r = _run(["-c", code])
    assert r.returncode == 0 and "late-converters-ok" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]


def test_shares_of_a_tile_that_are_given_up_are_summed_by_the_last_chunk():
    # a tile's first chunk is counted in 400000 cycles after the others, ten times what these wait for it before they give their shares of the rows up:
    # its CTA sums all rows.  Four shares and more, also where CTAs have several chunks; the counters are zero afterwards.
    code = textwrap.dedent("""
        import torch
        import paper_2402_02446_b200 as L
        dev = "cuda:0"
        g = torch.Generator(device=dev); g.manual_seed(10)
        draw = lambda *s: torch.randn(s, generator=g, device=dev)
        for K, N, n in ((11008, 264, 1), (4096, 4096, 1), (8192, 2424, 15)):
            Pg = L.prepare_weights(draw(K, N) * 0.02, draw(K, 40) / K ** 0.5, draw(40, N) * 0.01)
            for M, dtype in ((17, torch.float32), (49, torch.bfloat16), (128, torch.float32)):
                X = draw(M, K)
                Ys = [torch.full((M, N), float("nan"), dtype=dtype, device=dev) for _ in range(n)]
                calls = L.make_calls([(X, Pg, y) for y in Ys], torch.float32, dtype)
                ws = torch.zeros(L.batched_workspace_bytes(calls), dtype=torch.uint8, device=dev)
                L.linear_batched_ex(calls, ws, torch.float32, dtype)
                assert L.poll_status(ws) == 0
                want = [y.clone() for y in Ys]
                ws[168192:] = 0xFF
                L.debug_converter_lag(100_000)
                try:
                    L.linear_batched_ex(calls, ws, torch.float32, dtype)
                    assert L.poll_status(ws) == 0, (K, M)
                finally:
                    L.debug_converter_lag(0)
                assert all(torch.equal(y, w) for y, w in zip(Ys, want)), (K, M)
                L.linear_batched_ex(calls, ws, torch.float32, dtype)
                assert L.poll_status(ws) == 0 and all(torch.equal(y, w) for y, w in zip(Ys, want)), (K, M)
            Pg.release()
        print("given-up-ok")
    """)
    r = _run(["-c", code])
    assert r.returncode == 0 and "given-up-ok" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]


def test_weight_stages_that_land_late_lose_nothing():
    # the cluster kernel's ring (rings of 5, 4, 17 and 20 slots): every fifth stage from the second round on lands some 10 us after the others that
    # the ring has room for.  Whoever took the stage before it for its own would multiply that one's weights.
    code = textwrap.dedent("""
        import torch
        import paper_2402_02446_b200 as L
        dev = "cuda:0"
        g = torch.Generator(device=dev); g.manual_seed(8)
        draw = lambda *s: torch.randn(s, generator=g, device=dev)
        for M, K, N, k, w_bits in ((16, 11008, 11008, 32, 4), (16, 12288, 11008, 32, 4), (4, 4096, 20488, 32, 4), (8, 4096, 25096, 0, 2)):
            cfg = L.default_config(); cfg.w_bits = w_bits
            A, B = (draw(K, k) / K ** 0.5, draw(k, N) * 0.01) if k else (None, None)
            Pg = L.prepare_weights(draw(K, N) * 0.02, A, B, cfg)
            X = draw(M, K)
            ws = L.new_workspace(M, Pg)
            Y = L.linear(X, Pg, ws).clone()
            assert L.poll_status(ws) == 0
            L.debug_converter_lag(20_000)
            try:
                before = L.launch_count()
                late = L.linear(X, Pg, ws)
                assert L.launch_count() - before == 1
                assert L.poll_status(ws) == 0, (M, K)
            finally:
                L.debug_converter_lag(0)
            assert torch.equal(late, Y), (M, K)
            Pg.release()
        print("late-stages-ok")
    """)
    r = _run(["-c", code])
    assert r.returncode == 0 and "late-stages-ok" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]


def test_whoever_waits_for_the_clusters_that_form_t_in_vain_forms_it():
    # the cluster kernel under the same hook: T never counts as complete (as if its clusters waited for places that other launches hold), so every
    # warp that needs it forms it.  The sums are the same in the same order: Y is that of the ordinary call, and no wait runs out.
    code = textwrap.dedent("""
        import torch
        import paper_2402_02446_b200 as L
        dev = "cuda:0"
        g = torch.Generator(device=dev); g.manual_seed(9)
        draw = lambda *s: torch.randn(s, generator=g, device=dev)
        # one rank block to a cluster, two, six and more than warps are; one, two, four and eight CTAs that share K; a ragged last block of ranks
        for K, N, k, M, w_bits in ((1040, 20008, 40, 5, 4), (2112, 264, 256, 3, 4), (2048, 2048, 256, 16, 4), (4096, 1032, 130, 9, 4),
                                   (1040, 648, 136, 8, 2), (256, 4104, 200, 16, 4), (64, 4104, 36, 4, 4), (12288, 520, 200, 12, 4)):
            cfg = L.default_config(); cfg.w_bits = w_bits
            Pg = L.prepare_weights(draw(K, N) * 0.02, draw(K, k) / K ** 0.5, draw(k, N) * 0.01, cfg)
            # X of many binades: the fp64 sums round, so their order shows
            X = draw(M, K) * torch.exp2(torch.randint(-30, 31, (M, K // 16), generator=g, device=dev).float()).repeat_interleave(16, 1)
            for x in (X, X.bfloat16()):
                ws = L.new_workspace(M, Pg)
                Y = L.linear_ex(x, Pg, ws).clone()
                assert L.poll_status(ws) == 0
                L.debug_converter_lag(1)
                try:
                    before = L.launch_count()
                    alone = L.linear_ex(x, Pg, ws)
                    assert L.launch_count() - before == 1
                    assert L.poll_status(ws) == 0, (K, M)
                finally:
                    L.debug_converter_lag(0)
                assert torch.equal(alone, Y), (K, M, k)
                assert torch.equal(L.linear_ex(x, Pg, ws), Y) and L.poll_status(ws) == 0
            Pg.release()
        print("t-alone-ok")
    """)
    r = _run(["-c", code])
    assert r.returncode == 0 and "t-alone-ok" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]


def test_the_ordinary_build_has_no_such_hook():
    import paper_2402_02446_b200 as L
    from paper_2402_02446_b200 import binding
    if binding.DEBUG_BOUNDS:
        pytest.skip("this process runs the checked build")
    assert L.lib().lqer_debug_bounds_shrink(16) == binding.STATUS_NAMES.index("LQER_ERR_CONFIG")
    assert L.lib().lqer_debug_converter_lag(16) == binding.STATUS_NAMES.index("LQER_ERR_CONFIG")
