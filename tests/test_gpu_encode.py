"""The CUDA encoder back end against the host encoder: the same bytes for the same input, and therefore
(tests/test_library_host.py) the oracle's bytes as well."""
import os
import subprocess
import threading

import numpy as np
import pytest
import torch

import oracle
import paper_2609_34185_b200 as ep
from paper_2609_34185_b200 import synth
from test_encode_core import ROOT, disjoint_cosets

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("maker,shape,bpp,kw", [
    (synth.gaussian_rows, (512, 512), 4.0, dict(tile_vectors=4096)),
    (synth.laplace_rows, (96, 1024), 2.0, {}),
    (synth.student_t_rows, (256, 2048), 3.0, dict(tile_vectors=455)),
    (synth.laplace_rows, (64, 4096), 6.0, {}),
    (synth.gaussian_rows, (33, 264), 5.0, dict(tile_vectors=100)),
    (synth.gaussian_rows, (8, 8), 4.0, {}),
    (synth.gaussian_rows, (128, 1024), 8.0, {}),                    # b = 12
])
def test_device_encoder_gives_the_host_encoders_bytes(maker, shape, bpp, kw):
    W = maker(shape[0], shape[1], 4242 + shape[0])
    host = ep.encode(W, bpp, **kw)
    dev = ep.encode_device(torch.from_numpy(W).cuda(), bpp, **kw)
    assert np.array_equal(dev.data, host.data)
    assert dev.report["s"] == host.report["s"] and dev.report["b"] == host.report["b"]
    assert ep.validate(dev.data) == 0


def test_device_encoder_full_size_and_round_trip():
    W = synth.config2()
    Wd = torch.from_numpy(W).cuda()
    blob = ep.encode_device(Wd, 3.0)
    ref, rep = oracle.encode(W, 3.0)
    assert np.array_equal(blob.data, ref)
    out = ep.decode(ep.upload(blob), ep.BF16)
    torch.cuda.synchronize()
    e = oracle.rel_l2(W, out.float().cpu().numpy())
    assert 0.05 < e < 0.25 and abs(blob.stored_bpp - 3.0) < 0.03


def test_device_encoder_falls_back_cleanly_on_huge_coordinates():
    # one non-zero weight per row: the normalised value is sqrt(C) = 64, and with nothing else to code the search
    # runs to the fine end of its bracket (s = 1e-3), tens of thousands of lattice steps away from zero
    W = np.zeros((16, 4096), np.float32)
    W[np.arange(16), np.arange(16) * 5] = 1.0
    with pytest.raises(ep.EntroPackError) as ei:
        ep.encode_device(torch.from_numpy(W).cuda(), 8.0)
    assert ei.value.status == -3
    assert ep.validate(ep.encode(W, 8.0).data) == 0          # the host encoder still serves it


def test_device_encoder_leaves_the_per_row_refinement_to_the_host():
    W = synth.gaussian_rows(32, 512, 11)
    with pytest.raises(ep.EntroPackError) as ei:
        ep.encode_device(torch.from_numpy(W).cuda(), 4.0, rdo_candidates=3)
    assert ei.value.status == -3


def test_device_encoder_blobs_keep_their_bytes_while_buffers_are_reused():
    # finished blobs live in page-locked memory and a freed blob's buffer serves a later encode: a blob that is
    # still alive must never be overwritten, a reused buffer must give the same bytes as a fresh one
    import gc
    Wa, Wb = synth.gaussian_rows(256, 1024, 71), synth.laplace_rows(192, 2048, 72)
    da, db = torch.from_numpy(Wa).cuda(), torch.from_numpy(Wb).cuda()
    ref_a, ref_b = ep.encode(Wa, 4.0).data.copy(), ep.encode(Wb, 3.0).data.copy()
    a1 = ep.encode_device(da, 4.0)
    b1 = ep.encode_device(db, 3.0)                 # a1 alive: must come from another buffer
    assert np.array_equal(a1.data, ref_a) and np.array_equal(b1.data, ref_b)
    view = a1.data[100:200]
    keep = view.copy()
    del a1
    gc.collect()                                   # `view` still holds the buffer
    b2 = ep.encode_device(db, 3.0)
    assert np.array_equal(view, keep) and np.array_equal(b2.data, ref_b)
    del view, b1, b2
    gc.collect()
    for _ in range(3):                             # now buffers come back from the spare slot
        a = ep.encode_device(da, 4.0)
        assert np.array_equal(a.data, ref_a)
        del a
        gc.collect()
        b = ep.encode_device(db, 3.0)
        assert np.array_equal(b.data, ref_b)
        del b
        gc.collect()


def _wide_alphabet(magnitude):
    # a few outliers of up to `magnitude` row sigmas in every coordinate position stretch the tables
    W = synth.gaussian_rows(256, 2048, 5)
    rng = np.random.default_rng(5)
    sig = W.std(1)
    for i in range(400):
        r = rng.integers(256)
        W[r, rng.integers(2048)] = magnitude * sig[r] * (1 if i % 2 else -1) * rng.uniform(0.8, 1.0)
    return W


def _grid(R, C):
    # weights on a coarse grid, half the rows all zero: quantiser inputs on ties, where only the exact path decides
    W = np.round(synth.gaussian_rows(R, C, 6) * 64).astype(np.float32) / 64
    W[::2] = 0.0
    return W


@pytest.mark.parametrize("W,bpp,kw", [
    (_wide_alphabet(20.0), 6.0, {}),          # 7 k symbols: counts that take a second copy, wide code tables
    (_wide_alphabet(20.0), 8.0, {}),          # 20 k symbols
    (_wide_alphabet(40.0), 8.0, {}),          # over 25 k: a step the device hands to the host, tables in global memory
    (_grid(64, 1024), 3.0, {}),
    (_grid(5, 8), 2.0, {}),
    (synth.laplace_rows(1, 40960, 7), 4.0, dict(tile_vectors=33)),       # one long row, ragged tiles
    (synth.gaussian_rows(3000, 8, 8), 4.0, dict(polish_steps=0)),        # one block per row
    (synth.gaussian_rows(300, 1032, 9), 5.0, dict(search_steps=0)),
    (synth.gaussian_rows(300, 1032, 9), 5.0, dict(b_start=9, b_max=13, sample_vectors=500)),
])
def test_device_encoder_bytes_at_the_edges_of_its_paths(W, bpp, kw):
    host = ep.encode(W, bpp, **kw)
    dev = ep.encode_device(torch.from_numpy(np.ascontiguousarray(W, np.float32)).cuda(), bpp, **kw)
    assert np.array_equal(dev.data, host.data) and dev.report == host.report


def _outlier_rows(R, C, seed):
    return synth.gaussian_rows(R, C, seed, outlier_p=0.002)


@pytest.mark.parametrize("maker,shape,bpp,kw", [
    (synth.laplace_rows, (480, 1024), 6.0, {}),                    # steps of the search judged by the entropy of their counts
    (synth.laplace_rows, (480, 1024), 8.0, {}),                    # and alphabets whose excess of slots takes hundreds of turns
    (synth.laplace_rows, (480, 1024), 8.0, dict(b_start=11, b_max=11)),
    (_outlier_rows, (64, 4096), 8.0, {}),
    (_outlier_rows, (512, 1024), 7.0, dict(polish_steps=0)),
])
def test_device_encoder_bytes_with_wide_alphabets(maker, shape, bpp, kw):
    W = maker(*shape, 12)
    host = ep.encode(W, bpp, **kw)
    dev = ep.encode_device(torch.from_numpy(W).cuda(), bpp, **kw)
    assert np.array_equal(dev.data, host.data) and dev.report == host.report


@pytest.mark.parametrize("bpp", [8.0, 2.0])
def test_device_encoder_bytes_with_cosets_that_do_not_meet(bpp):
    W = disjoint_cosets()
    host = ep.encode(W, bpp)
    dev = ep.encode_device(torch.from_numpy(W).cuda(), bpp)
    assert np.array_equal(dev.data, host.data) and dev.report == host.report


@pytest.mark.timeout(60)
@pytest.mark.parametrize("maker,bpp,steps", [
    (synth.gaussian_rows, 4.0, 2**31 - 1),        # as many corrections as it takes, which are few
    (synth.laplace_rows, 6.0, 1000),
    (synth.laplace_rows, 6.0, 7),                 # the last pass before the device is asked whether it has stopped
    (synth.laplace_rows, 6.0, 8),
])
def test_device_encoder_with_any_number_of_rate_corrections(maker, bpp, steps):
    W = maker(64, 1024, 21)
    host = ep.encode(W, bpp, polish_steps=steps)
    dev = ep.encode_device(torch.from_numpy(W).cuda(), bpp, polish_steps=steps)
    assert np.array_equal(dev.data, host.data) and dev.report == host.report


@pytest.mark.parametrize("shape,V", [
    ((128, 1024), 16),            # 1024 tiles: one turn of the last CTA's prefix sum
    ((129, 1024), 16),            # and eight more
    ((370, 1024), 16),            # 2960 tiles, the last number of four-warp CTAs
    ((371, 1024), 16),            # eight warps per CTA
    ((592, 1024), 16),            # 4736 tiles, their last number
    ((593, 1024), 16),            # sixteen
    ((64, 8), 1),                 # tiles of one block
])
def test_device_encoder_bytes_by_number_of_tiles(shape, V):
    W = synth.gaussian_rows(*shape, 31)
    host = ep.encode(W, 4.0, tile_vectors=V)
    dev = ep.encode_device(torch.from_numpy(W).cuda(), 4.0, tile_vectors=V)
    assert np.array_equal(dev.data, host.data) and dev.report == host.report


def test_device_encoder_codes_again_where_the_host_moves_on():
    # sampled rows with few distinct coordinates, the others Laplacian: the scale found on the sample gives the full tensor alphabets that
    # do not fit, so the host goes to the next precision or, at the highest, to coarser scales of its own
    R, C, budget = 128, 4096, 1 << 13
    rows = oracle.sample_rows(R, C, budget)
    W = synth.laplace_rows(R, C, 44)
    W[rows] = np.random.Generator(np.random.PCG64(45)).uniform(-0.02, 0.02, (len(rows), C)).astype(np.float32)
    Wd, moved = torch.from_numpy(W).cuda(), set()
    for kw in (dict(b_max=9), dict(b_max=9, polish_steps=0), dict(b_max=12)):
        host = ep.encode(W, 9.0, sample_vectors=budget, b_start=9, **kw)
        dev = ep.encode_device(Wd, 9.0, sample_vectors=budget, b_start=9, **kw)
        assert np.array_equal(dev.data, host.data) and dev.report == host.report
        moved.add(host.report["b"])
    assert len(moved) == 2


def test_device_encoder_bytes_with_several_encodes_at_once():
    # CTAs of one call's passes start late where another call holds the SMs: two threads, each with a stream and a workspace of its own
    jobs = [[(synth.gaussian_rows(256, 2048, 91), 4.0, {}), (synth.laplace_rows(64, 4096, 92), 6.0, dict(search_steps=9))],
            [(synth.student_t_rows(700, 1032, 93), 3.0, dict(sample_vectors=3000)), (synth.gaussian_rows(1024, 4096, 94), 5.0, {})]]
    refs = [[ep.encode(W, bpp, **kw).data for W, bpp, kw in mine] for mine in jobs]
    devs = [[torch.from_numpy(W).cuda() for W, _, _ in mine] for mine in jobs]
    workspaces = [torch.empty(max(W.size for W, _, _ in mine) * 8 + (16 << 20), dtype=torch.uint8, device="cuda") for mine in jobs]
    streams, wrong, failed = [torch.cuda.Stream() for _ in jobs], [], []
    torch.cuda.synchronize()

    def work(t):
        torch.cuda.set_device(devs[t][0].device)
        try:
            for turn in range(40):
                for i, (_, bpp, kw) in enumerate(jobs[t]):
                    got = ep.encode_device(devs[t][i], bpp, workspace=workspaces[t], stream=streams[t], **kw)
                    if not np.array_equal(got.data, refs[t][i]):
                        wrong.append((t, i, turn))
        except ep.EntroPackError as e:
            failed.append((t, e))

    threads = [threading.Thread(target=work, args=(t,)) for t in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong and not failed


def test_device_encoder_ends_searches_that_meet_scales_without_tables(tmp_path):
    # the target is above what the finest scale with a table gives, so the last steps of a search often find no table: the
    # counts of the last step that had one are of an earlier pass
    exe, csrc = str(tmp_path / "search_done"), os.path.join(ROOT, "paper_2609_34185_b200", "csrc")
    nvcc = os.environ.get("NVCC") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-O1", "-std=c++17", "-Xcompiler", "-ffp-contract=off,-pthread",
                    "-I", os.path.join(ROOT, "include"), "-I", csrc, "-o", exe, os.path.join(ROOT, "tests", "search_done.cu")]
                   + [os.path.join(csrc, f) for f in ("encoder.cpp", "stream.cpp")], check=True)
    Ws = [synth.laplace_rows(96, 1024, 700 + i) for i in range(24)]
    np.stack(Ws).tofile(tmp_path / "w.bin")
    run = subprocess.run([exe, str(tmp_path / "w.bin"), "24", "96", "1024", "12.0", "9"], check=True, capture_output=True, text=True, timeout=60)
    assert run.stdout.split() == ["1"] * 24
    for W in Ws[:6]:
        host = ep.encode(W, 12.0, b_start=9, b_max=9, polish_steps=0)
        dev = ep.encode_device(torch.from_numpy(W).cuda(), 12.0, b_start=9, b_max=9, polish_steps=0)
        assert np.array_equal(dev.data, host.data) and dev.report == host.report


@pytest.mark.parametrize("shape", [(64, 1024), (1100, 1024)])        # up to fifteen scales per pass; more than 2^17 blocks: nine
@pytest.mark.parametrize("bpp,kw", [
    (4.0, dict(search_steps=1)),
    (4.0, dict(search_steps=2)),
    (4.0, dict(search_steps=3)),
    (4.0, dict(search_steps=4)),
    (4.0, dict(search_steps=7)),
    (4.0, dict(search_steps=14)),
    (4.0, dict(search_steps=60)),                                     # the bracket's ends meet
    (4.0, dict(bracket_lo=0.2, bracket_hi=0.3)),
    (4.0, dict(bracket_lo=0.25, bracket_hi=0.25000001)),              # the same scale all the way
    (3.0, dict(bracket_lo=0.05, bracket_hi=0.1)),                     # the target is on one side of the bracket: one-sided forecasts to the end,
    (6.0, dict(bracket_lo=0.5, bracket_hi=2.0)),
    (6.0, dict(bracket_lo=0.5, bracket_hi=2.0, polish_steps=0)),
    (12.0, dict(b_start=9, b_max=9, polish_steps=0)),                 # beyond every scale with a table: trees of four steps
    (12.0, dict(b_start=9, b_max=9, polish_steps=0, search_steps=6)),
])
def test_device_encoder_searches_like_the_hosts(shape, bpp, kw):
    W = synth.laplace_rows(*shape, 77)
    host = ep.encode(W, bpp, **kw)
    dev = ep.encode_device(torch.from_numpy(W).cuda(), bpp, **kw)
    assert np.array_equal(dev.data, host.data) and dev.report == host.report
