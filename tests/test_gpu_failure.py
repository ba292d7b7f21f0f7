"""Failure detection on the GPU without a fault: a bounded wait that runs out.

The library's TMA pipelines bound every mbarrier wait; a wait that runs out sets a sticky
device flag and the kernel ends normally.  The self-test kernel drives that same path with
a small poll limit on an mbarrier that nothing arrives on, and the host reads the status;
afterwards the context must still run the hot path.

The GEMM kernels are built once more with one block whose epilogue gives up at once on its
accumulators (and a poll limit of some milliseconds for the waits that then run out too): the flag is
set, what the block owed is NaN, the other blocks' results are what they were, and the block has
waited for its own loads and MMAs, so nothing is in flight when it ends.
"""
import concurrent.futures as cf
import ctypes
import subprocess

import pytest
import torch

import paper_2608_28113_gb300 as hs
from paper_2608_28113_gb300 import build as cuda_build
from paper_2608_28113_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hs.load()


def test_bounded_wait_runs_out_reports_and_the_context_survives():
    dev = torch.device("cuda", 0)
    hs.hscale_device_error_flags()                      # start from a clean state
    for polls in (0, 1000):
        hs.hscale_selftest_bounded_wait(polls)
        torch.cuda.synchronize()
        assert hs.hscale_device_error_flags() & 1, f"timeout not reported ({polls} polls)"
        assert hs.hscale_device_error_flags() == 0      # the flags clear on read
    x = torch.ones(256, 64, dtype=torch.bfloat16, device=dev) * 2
    h = torch.zeros(64, dtype=torch.float32, device=dev)
    hs.hscale_hessian_diag_accumulate(x, h)
    torch.cuda.synchronize()
    assert torch.all(h == 256 * 4.0)
    assert hs.hscale_device_error_flags() == 0


# ---------------------------------------------------------------- the GEMM kernels' waits
@pytest.fixture(scope="module", params=[0, 1])
def starved(request, tmp_path_factory):
    """(block, library): the library built with that starved block."""
    block, out = request.param, tmp_path_factory.mktemp("starved")

    def compile_one(src):
        obj = out / (src.stem + ".o")
        subprocess.run([cuda_build.nvcc_path(), *cuda_build.ARCH, *cuda_build.NVCC_FLAGS,
                        f"-DHSCALE_STARVED_BLOCK={block}", "-c", str(src), "-o", str(obj)], check=True,
                       capture_output=True)
        return str(obj)

    with cf.ThreadPoolExecutor(8) as ex:
        objs = list(ex.map(compile_one, cuda_build.sources()))
    so = out / f"libhscale_starved{block}.so"
    subprocess.run([cuda_build.nvcc_path(), *cuda_build.ARCH, "-shared", "-o", str(so), *objs], check=True)
    lib = ctypes.CDLL(str(so))
    for name, (res, args) in hs._SIGNATURES.items():
        fn = getattr(lib, name)
        fn.restype, fn.argtypes = res, args
    return block, lib


def both(starved, monkeypatch, call):
    """call() under the starved library, whose flag it must set, then under the real one, whose flag
    stays clear."""
    hs.hscale_device_error_flags()
    with monkeypatch.context() as patch:
        patch.setattr(hs, "_lib", starved[1])
        got = call()
        torch.cuda.synchronize()
        assert hs.hscale_device_error_flags() == 1
        assert hs.hscale_device_error_flags() == 0
    want = call()
    torch.cuda.synchronize()
    assert hs.hscale_device_error_flags() == 0
    return got, want


def activations(tokens, n, lead=0):
    g = torch.Generator(device="cuda").manual_seed(tokens + n)
    return torch.randn(tokens, n + lead, generator=g, device="cuda").to(torch.bfloat16)[:, lead:]


@pytest.mark.parametrize("lead", [0, 1])  # X as it is, and transposed first
def test_full_hessian_tile_of_a_starved_block(starved, monkeypatch, lead):
    x = activations(5000, 768, lead)  # three segments, one CTA a tile

    def call():
        H = torch.zeros(768, 768, device="cuda")
        hs.hscale_hessian_full_accumulate(x, H)
        return H

    got, want = both(starved, monkeypatch, call)
    tile = torch.zeros_like(want, dtype=torch.bool)
    tile[:128, 256 * starved[0]:256 * starved[0] + 256] = True
    assert bool(torch.isnan(got[tile]).all()) and torch.equal(got[~tile], want[~tile])


@pytest.mark.parametrize("tokens,n", [(9000, 2000), (8192, 384), (18000, 130)])  # clusters of 2, 4 and 8
def test_full_hessian_tile_of_a_starved_rank(starved, monkeypatch, tokens, n):
    """The starved block is one rank of the first tile's cluster.  The others add its partial to their
    columns, so none of the tile's values stands."""
    x = activations(tokens, n)

    def call():
        H = torch.zeros(n, n, device="cuda")
        hs.hscale_hessian_full_accumulate(x, H)
        return H

    got, want = both(starved, monkeypatch, call)
    tile = torch.zeros_like(want, dtype=torch.bool)
    tile[:128, :256] = True
    assert bool(torch.isnan(got[tile]).all()) and torch.equal(got[~tile], want[~tile])


def test_output_error_of_a_starved_block(starved, monkeypatch):
    x, dw2 = activations(300, 2048), activations(512, 4096)
    ws = torch.empty(hs.hscale_output_error_workspace_bytes(300, 512), dtype=torch.uint8, device="cuda")

    def call():
        out = torch.zeros(1, dtype=torch.float64, device="cuda")
        hs.hscale_output_error(x, dw2, 512, out, ws)
        return out

    got, want = both(starved, monkeypatch, call)
    assert bool(torch.isnan(got)) and bool(torch.isfinite(want))


def test_factor_with_a_starved_block(starved, monkeypatch):
    """Block 0 owes the next diagonal block, whose pivots then fail; block 1 the first tile of the
    update, whose NaN reach U.  The sweep ends either way."""
    x = activations(2048, 640).float()
    H = (x.T @ x).contiguous()

    def call():
        U, info = torch.zeros(640, 640, device="cuda"), torch.zeros(3, dtype=torch.int32, device="cuda")
        hs.hscale_gptq_factor(H, 0.01, U, None, info)
        return U, info

    (U, info), (Uw, infow) = both(starved, monkeypatch, call)
    assert bool(torch.isnan(U).any()) or info[0].item() > 0
    assert bool(torch.isfinite(Uw).all()) and infow[0].item() == 0


def test_block_loop_with_a_starved_block(starved, monkeypatch):
    """The first panel is starved in rows 16 b .. 16 b + 15 from its second block on, so its other codes
    are what they were; the update's NaN come after it."""
    m, n, block = 64, 1024, 128
    w = wl.weight(m, n, 0.02, 5, torch.device("cuda"))
    U = torch.triu(torch.randn(n, n, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda") * 0.01)
    U.fill_diagonal_(1.0)
    h, sg = torch.ones(n, device="cuda"), torch.full((1,), 3e-5, device="cuda")

    def call():
        codes = torch.zeros(m, n // 16, dtype=torch.uint8, device="cuda")
        packed = torch.zeros(m, n // 2, dtype=torch.uint8, device="cuda")
        hs.hscale_gptq_hscale(w, U, h, sg, None, block, 4, 4, codes, packed)
        return codes[:, :512 // 16], packed[:, :512 // 2]

    got, want = both(starved, monkeypatch, call)
    rows = torch.ones(m, dtype=torch.bool, device="cuda")
    rows[16 * starved[0]:16 * starved[0] + 16] = False
    for g, v in zip(got, want):
        assert torch.equal(g[rows], v[rows])
        assert torch.equal(g[:, :v.shape[1] // 4], v[:, :v.shape[1] // 4])
