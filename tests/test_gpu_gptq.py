"""GPU parity of GPTQ + H-Scale (Algorithm 3) against the fp64 CPU oracle.

Pass rules:
  * H = X^T X on the tensor cores: |H_gpu - H| <= 1e-5 * sqrt(H_ii H_jj) (bf16 products are
    exact; fp32 accumulation over the tokens).
  * the factor U (the library's blocked fp32 Cholesky of the reversed 1 %-damped H and its
    triangular inverse, updates on the tensor cores in three-way bf16 splits): relative Frobenius error
    <= 1e-3 against numpy's fp64 factor of the same fp32 H; identical dead channels.
  * the block loop, fed the same fp32 U, h and s_g as the oracle: the first block's codes and
    nibbles bit-exact outside the oracle's near-ties; one block (B = n) and a diagonal U (no
    propagation) bit-exact outside near-ties; with propagation the fp32 running weights
    drift from the oracle's fp64 ones, so later blocks are checked through >= 98 % equal
    codes and the layer-output error ||X dW^T||^2 of the result within 1 %.
"""
import os

import numpy as np
import pytest
import torch

import oracle
import paper_2608_28113_gb300 as hs
from paper_2608_28113_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hs.load()
    oracle.set_threads(os.cpu_count() or 1)


def dev():
    return torch.device("cuda", 0)


def bits(t):
    return wl.bf16_bits(t)


def calib(n, tokens, seed):
    a = wl.channel_magnitudes(n, 1.0, 4, 50.0, seed)
    return wl.activation_chunk(tokens, a, seed, 0)


def oracle_H(x, n):
    H = np.zeros((n, n))
    oracle.hessian_full(bits(x), H)
    return H


@pytest.mark.parametrize("tokens,n,chunks,view", [(128, 256, 1, "whole"), (300, 200, 1, "whole"),
                                                  (1000, 520, 2, "whole"), (77, 131, 1, "whole"),
                                                  (200, 96, 2, "aligned slice"), (150, 72, 1, "odd slice"),
                                                  (4500, 136, 1, "whole"), (9000, 264, 2, "whole"),
                                                  (65536, 256, 1, "whole")])
def test_full_hessian_matches_oracle(tokens, n, chunks, view):
    """Whole X, a ragged width (n % 8 != 0), a 16-byte aligned column slice of a wider X
    (ld_x > n) and a slice starting at an odd column (the 2-byte transpose path); calls
    of several 2048-token accumulation segments with a ragged last one; and one call of
    65536 tokens, whose error stays that of a 2048-token segment (one long fp32
    accumulation on the tensor cores would be 30x over the bound there)."""
    x = calib(n, tokens, 60 + n)
    ref = oracle_H(x, n)
    if view == "whole":
        xd = x.to(dev())
    else:
        off = 8 if view == "aligned slice" else 1
        wide = torch.zeros(tokens, n + 24, dtype=torch.bfloat16, device=dev())
        wide[:, off:off + n] = x.to(dev())
        xd = wide[:, off:off + n]
    H = torch.zeros(n, n, dtype=torch.float32, device=dev())
    step = (tokens + chunks - 1) // chunks
    for t0 in range(0, tokens, step):
        hs.hscale_hessian_full_accumulate(xd[t0:t0 + step], H)
    torch.cuda.synchronize()
    got = H.cpu().double().numpy()
    scale = np.sqrt(np.outer(np.diag(ref), np.diag(ref)))
    err = np.triu(np.abs(got - ref))        # the upper triangle is the accumulated part
    assert np.all(err <= 1e-5 * scale + 1e-30), f"max scaled err {np.max(err / (scale + 1e-300)):.2e}"
    assert hs.hscale_device_error_flags() == 0


@pytest.mark.parametrize("tokens,n,view", [
    (8192, 256, "whole"),            # four segments: clusters of four
    (8193, 384, "whole"),            # a fifth of one token
    (18000, 130, "whole"),           # nine segments in clusters of eight; unaligned H rows, K-major operands
    (10240, 1280, "aligned slice"),  # five segments, clusters of four; widths past one tile
    (9000, 2000, "whole"),           # clusters of two; n not a multiple of 64
    (4100, 1001, "whole"),           # two full segments and a third, unaligned rows
])
def test_full_hessian_by_clusters(tokens, n, view):
    """Widths whose tiles are split over a cluster's CTAs: into an H that is not zero, a call adds
    the sum of its 2048-token segments, bit for bit that of calls of one segment each into a
    zeroed H; only the tiles on and above the diagonal are written."""
    x = calib(n, tokens, 300 + n).to(dev())
    if view == "aligned slice":
        wide = torch.zeros(tokens, n + 24, dtype=torch.bfloat16, device=dev())
        wide[:, 8:8 + n] = x
        x = wide[:, 8:8 + n]
    H1 = torch.zeros(n, n, dtype=torch.float32, device=dev())
    H2 = torch.zeros_like(H1)
    base = torch.full((n, n), 3.0, dtype=torch.float32, device=dev())
    H3 = base.clone()
    hs.hscale_hessian_full_accumulate(x, H1)
    hs.hscale_hessian_full_accumulate(x, H3)
    for t0 in range(0, tokens, 2048):
        hs.hscale_hessian_full_accumulate(x[t0:t0 + 2048], H2)
    torch.cuda.synchronize()
    i = torch.arange(n, device=dev())
    written = (i[None, :] // 256 + 1) * 256 > (i[:, None] // 128) * 128
    assert torch.equal(H1[written], H2[written]) and bool((H1[~written] == 0).all())
    assert torch.equal(H3[written], (base + H2)[written]) and bool((H3[~written] == 3).all())
    d = torch.diagonal(H1).double()
    ref = x.double().square().sum(0)
    assert bool(((d - ref).abs() <= 1e-5 * ref + 1e-30).all())
    assert hs.hscale_device_error_flags() == 0


def test_full_hessian_one_call_equals_2048_token_calls():
    """The kernel's accumulation segments: one call over 12,000 tokens gives, bit for bit,
    the H of successive calls of 2048 tokens (the last one ragged)."""
    n, tokens = 384, 12000
    x = calib(n, tokens, 91).to(dev())
    H1 = torch.zeros(n, n, dtype=torch.float32, device=dev())
    H2 = torch.zeros_like(H1)
    hs.hscale_hessian_full_accumulate(x, H1)
    for t0 in range(0, tokens, 2048):
        hs.hscale_hessian_full_accumulate(x[t0:t0 + 2048], H2)
    torch.cuda.synchronize()
    assert torch.equal(torch.triu(H1), torch.triu(H2))
    assert hs.hscale_device_error_flags() == 0


def gpu_factor(H32, damp=0.01):
    n = H32.shape[0]
    U = torch.empty(n, n, dtype=torch.float32, device=dev())
    dead = torch.empty(n, dtype=torch.uint8, device=dev())
    info = torch.full((3,), -7, dtype=torch.int32, device=dev())
    hs.hscale_gptq_factor(torch.from_numpy(H32).to(dev()), damp, U, dead, info)
    torch.cuda.synchronize()
    return U.cpu().double().numpy(), dead.cpu().numpy().astype(bool), info.cpu().numpy()


def test_factor_matches_oracle_with_a_dead_channel():
    n = 256
    x = calib(n, 512, 71)
    x[:, 17] = 0
    H32 = oracle_H(x, n).astype(np.float32)
    U, dead, info = gpu_factor(H32)
    Uref, dref = oracle.gptq_factor(H32.astype(np.float64))
    assert np.all(info == 0), info
    assert np.array_equal(dead, dref) and dead[17] and dead.sum() == 1
    assert np.all(np.tril(U, -1) == 0)
    rel = np.linalg.norm(U - Uref) / np.linalg.norm(Uref)
    print(f"[parity] gptq factor n={n}: rel Frobenius err {rel:.2e}")
    assert rel <= 1e-3


@pytest.mark.parametrize("n,tokens", [(72, 300), (128, 400), (131, 500), (200, 600), (384, 1200), (1000, 3000)])
def test_factor_sizes_across_block_boundaries(n, tokens):
    """Widths below one 128-wide block, exactly one, ragged (padded with an identity block) and
    several blocks (trailing and inverse updates on the tensor cores)."""
    x = calib(n, tokens, 700 + n)
    H32 = oracle_H(x, n).astype(np.float32)
    U, dead, info = gpu_factor(H32)
    Uref, dref = oracle.gptq_factor(H32.astype(np.float64))
    assert np.all(info == 0), info
    assert np.array_equal(dead, dref)
    assert np.all(np.tril(U, -1) == 0)
    rel = np.linalg.norm(U - Uref) / np.linalg.norm(Uref)
    print(f"[parity] gptq factor n={n}: rel Frobenius err {rel:.2e}")
    assert rel <= 1e-4
    assert hs.hscale_device_error_flags() == 0


@pytest.mark.parametrize("power", [-104, 90])
def test_factor_of_a_scaled_matrix(power):
    """U of 2^power H is 2^(-power/2) U.  At these powers the pivots leave the range of the quick
    form of the diagonal blocks (2^-50 to 2^50), so their full-range form runs; both
    forms are within about 2^-22, and the factor's error grows with the condition of the damped H,
    so the bound is that of the oracle comparison above."""
    n = 300
    x = calib(n, 900, 17)
    H32 = oracle_H(x, n).astype(np.float32)
    U, dead, info = gpu_factor(H32)
    Us, deads, infos = gpu_factor(np.ldexp(H32, power).astype(np.float32))
    assert np.all(info == 0) and np.all(infos == 0) and np.array_equal(dead, deads)
    d = np.ldexp(Us, power // 2) - U
    assert np.linalg.norm(d) <= 1e-4 * np.linalg.norm(U)


@pytest.mark.parametrize("n", [128, 257, 640, 1000])
def test_factor_keeps_fp32_accuracy(n):
    """Sixteen tokens a channel: the condition of the damped H is small, so the factor's distance from
    64 bits is that of its arithmetic: 7e-8 measured, about a unit of fp32; the bound is four times
    that, where losing one of the products of the split operands would cost 2^-17 or more."""
    x = calib(n, 16 * n, 900 + n)
    H32 = oracle_H(x, n).astype(np.float32)
    U, _, info = gpu_factor(H32)
    Uref, _ = oracle.gptq_factor(H32.astype(np.float64))
    assert np.all(info == 0)
    rel = np.linalg.norm(U - Uref) / np.linalg.norm(Uref)
    print(f"[parity] gptq factor n={n}, 16 n tokens: rel Frobenius err {rel:.2e}, worst entry "
          f"{np.max(np.abs(U - Uref) / np.sqrt(np.outer(np.diag(Uref), np.diag(Uref)))):.2e}")
    assert rel <= 3e-7


def test_factor_of_a_14336_wide_layer():
    """n = 14,336 (an MLP's down projection): U^T U A v = v for the damped A, in 64 bits.  7e-7
    measured, U's own error times the condition of A; the bound is four times that."""
    n = 14336
    g = torch.Generator(device=dev()).manual_seed(3)
    x = torch.randn(2 * n, n, generator=g, device=dev())
    H = x.T @ x
    del x
    U = torch.empty(n, n, device=dev())
    info = torch.full((3,), -7, dtype=torch.int32, device=dev())
    hs.hscale_gptq_factor(H, 0.01, U, None, info)
    v = torch.randn(n, 4, generator=g, device=dev(), dtype=torch.float64)
    d = torch.diagonal(H).double()
    damp = 0.01 * d.mean()

    def times(M, y, transposed=False, sym=False):  # upper triangular M, row blocks at 64 bits
        out = torch.zeros(n, 4, dtype=torch.float64, device=dev())
        for r in range(0, n, 2048):
            b = torch.triu(M[r:r + 2048].double(), r)
            if sym or not transposed:
                out[r:r + 2048] += b @ y
            if sym or transposed:
                t = torch.triu(b, r + 1) if sym else b
                out += t.T @ y[r:r + 2048]
        return out

    z = times(U, times(U, times(H, v, sym=True) + damp * v), transposed=True)
    rel = float((z - v).norm() / v.norm())
    print(f"[parity] gptq factor n={n}: |U^T U A v - v| / |v| {rel:.2e}")
    assert info.cpu().tolist() == [0, 0, 0]
    assert bool((torch.tril(U, -1) == 0).all())
    assert rel <= 3e-6
    assert hs.hscale_device_error_flags() == 0


def test_factor_reports_a_matrix_that_is_not_positive_definite():
    """A symmetric matrix with a negative eigenvalue that the damping does not lift: info[0]
    names a failed pivot (1-based, in the reversed order); U is then unspecified."""
    n = 300
    rng = np.random.default_rng(5)
    Q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    ev = np.linspace(1.0, 2.0, n)
    ev[7] = -50.0
    H32 = ((Q * ev) @ Q.T).astype(np.float32)
    U, dead, info = gpu_factor(H32)
    assert 1 <= info[0] <= n and info[1] == 0 and info[2] == 0


@pytest.mark.parametrize("order", [1, 2, 15, 16, 17, 33, 128, 129, 250])
def test_factor_names_the_failed_pivot(order):
    """Near the identity (off-diagonal sums below 0.5, so every other pivot stays positive) with one
    entry at -5: the failed pivot is that entry, wherever it lies in its 2 x 2, 16 x 16 and 128 x 128
    block, and the sweep still ends with finite values."""
    n = 250
    noise = np.random.default_rng(order).uniform(-1e-3, 1e-3, (n, n))
    H = np.eye(n) + noise + noise.T
    H[n - order, n - order] = -5.0
    U, dead, info = gpu_factor(H.astype(np.float32))
    assert list(info) == [order, 0, 0]
    assert np.isfinite(U).all()


def gpu_gptq(w, U32, h32, s_g, block, down, up, dead=None, workspace=None):
    m, n = w.shape
    codes = torch.empty(m, n // 16, dtype=torch.uint8, device=dev())
    packed = torch.empty(m, n // 2, dtype=torch.uint8, device=dev())
    sg = torch.tensor([s_g], dtype=torch.float32, device=dev())
    dd = None if dead is None else torch.from_numpy(dead.astype(np.uint8)).to(dev())
    hs.hscale_gptq_hscale(w.to(dev()), torch.from_numpy(np.ascontiguousarray(U32)).to(dev()),
                          torch.from_numpy(h32).to(dev()), sg, dd, block, down, up, codes, packed, workspace)
    torch.cuda.synchronize()
    return codes.cpu().numpy(), packed.cpu().numpy()


def exact_outside_near_ties(codes, packed, ref, label):
    nt = ref["near_tie"].astype(bool)
    m, ng = codes.shape
    bad = (codes != ref["codes"]) & ~nt
    badp = (packed.reshape(m, ng, 8) != ref["packed"].reshape(m, ng, 8)).any(axis=2) & ~nt
    assert not bad.any() and not badp.any(), f"{label}: {bad.sum()} code / {badp.sum()} nibble mismatches"


def layer_inputs(m, n, seed, tokens=512):
    w = wl.weight(m, n, 0.02, seed)
    x = calib(n, tokens, seed + 1)
    H = oracle_H(x, n)
    U, dead = oracle.gptq_factor(H)
    return w, x, H, U.astype(np.float32), np.diag(H).astype(np.float32), dead


@pytest.mark.parametrize("block,window", [(64, (4, 4)), (32, (9, 6))])
def test_gptq_block_loop_matches_oracle(block, window):
    m, n = 96, 256
    w, x, H, U32, h32, dead = layer_inputs(m, n, 80 + block)
    wb = bits(w)
    s_g, _ = oracle.global_scale(wb)
    codes, packed = gpu_gptq(w, U32, h32, s_g, block, *window)
    ref = oracle.gptq_hscale(wb, U32.astype(np.float64), h32, s_g, block, *window, dead=dead)
    nb = block // 16
    first = {k: ref[k][:, :nb] for k in ("codes", "near_tie")}
    first["packed"] = ref["packed"][:, :block // 2]
    exact_outside_near_ties(codes[:, :nb], packed[:, :block // 2], first, "first block")
    agree = float(np.mean(codes == ref["codes"]))
    xe = x.float().double().numpy()
    e_gpu = oracle.output_error(xe, oracle.dequant_residual(wb, s_g, codes, packed))
    e_ref = oracle.output_error(xe, oracle.dequant_residual(wb, s_g, ref["codes"], ref["packed"]))
    print(f"[parity] gptq {m}x{n} block {block} window {window}: codes equal {agree:.2%}, "
          f"output error gpu {e_gpu:.6e} oracle {e_ref:.6e}")
    assert agree >= 0.98
    assert abs(e_gpu - e_ref) <= 0.01 * e_ref


def test_gptq_one_block_and_diagonal_factor_reduce_to_the_search():
    m, n = 64, 128
    w, x, H, U32, h32, dead = layer_inputs(m, n, 90)
    wb = bits(w)
    s_g, _ = oracle.global_scale(wb)
    ref = oracle.refine(wb, h32, s_g, None, 4, 4)
    codes, packed = gpu_gptq(w, U32, h32, s_g, n, 4, 4)
    exact_outside_near_ties(codes, packed, ref, "one block")
    Ud = np.diag(np.diag(U32)).astype(np.float32)
    codes, packed = gpu_gptq(w, Ud, h32, s_g, 16, 4, 4)
    exact_outside_near_ties(codes, packed, ref, "diagonal factor")


@pytest.mark.parametrize("m,n,block", [
    (1, 64, 16),        # one row; four blocks in one panel
    (33, 1104, 48),     # panels of 480 columns and a ragged last one; rows of three CTAs, the last ragged
    (17, 528, 16),      # a last panel of a single block
    (40, 768, 256),     # the widest block with an update inside the panel
    (24, 1024, 512),    # a block per panel
    (20, 1152, 576),    # a block wider than a panel
    (2448, 256, 64),    # more than 16 rows per SM: 32 rows a CTA
])
def test_gptq_panel_shapes(m, n, block):
    """Panel, block and row counts where the block loop's kernels change shape, against the
    oracle, under the rules above."""
    w, x, H, U32, h32, dead = layer_inputs(m, n, 500 + block, tokens=2 * n)
    wb = bits(w)
    s_g, _ = oracle.global_scale(wb)
    codes, packed = gpu_gptq(w, U32, h32, s_g, block, 4, 4, dead=dead)
    ref = oracle.gptq_hscale(wb, U32.astype(np.float64), h32, s_g, block, 4, 4, dead=dead)
    nb = block // 16
    first = {k: ref[k][:, :nb] for k in ("codes", "near_tie")}
    first["packed"] = ref["packed"][:, :block // 2]
    exact_outside_near_ties(codes[:, :nb], packed[:, :block // 2], first, "first block")
    assert float(np.mean(codes == ref["codes"])) >= 0.98
    assert hs.hscale_device_error_flags() == 0


@pytest.mark.parametrize("m,n,block", [(33, 1024, 16), (20, 1104, 48), (65, 1088, 64), (17, 1024, 128)])
def test_gptq_workspace_of_four_blocks(m, n, block):
    """The smallest workspace: m n floats and 12 block bf16 for each row of W and U.  The call takes it
    in panels of at most four blocks, touches nothing beyond it and agrees with the oracle under the
    rules above; one byte less is refused."""
    up256 = lambda b: (b + 255) // 256 * 256
    least = up256(4 * m * n) + up256(24 * block * m) + up256(24 * block * n)
    assert least <= hs.hscale_gptq_workspace_bytes(m, n, block)
    w, x, H, U32, h32, dead = layer_inputs(m, n, 600 + block, tokens=2 * n)
    wb = bits(w)
    s_g, _ = oracle.global_scale(wb)
    buf = torch.full((least + 4096,), 0xEE, dtype=torch.uint8, device=dev())
    with pytest.raises(hs.HScaleError):
        gpu_gptq(w, U32, h32, s_g, block, 4, 4, dead=dead, workspace=buf[:least - 1])
    codes, packed = gpu_gptq(w, U32, h32, s_g, block, 4, 4, dead=dead, workspace=buf[:least])
    assert bool((buf[least:] == 0xEE).all())
    ref = oracle.gptq_hscale(wb, U32.astype(np.float64), h32, s_g, block, 4, 4, dead=dead)
    assert float(np.mean(codes == ref["codes"])) >= 0.98
    full, _ = gpu_gptq(w, U32, h32, s_g, block, 4, 4, dead=dead)
    assert float(np.mean(codes == full)) >= 0.98
    assert hs.hscale_device_error_flags() == 0


@pytest.mark.parametrize("m,n", [(1300, 4096), (300, 4224), (2500, 1920)])
def test_gptq_rows_do_not_depend_on_the_others(m, n):
    """The update's last round of tiles may be halved, by how many there are, so by m; every
    element's products are summed in one order all the same: a call on some of the rows gives the
    bytes of the call on all of them."""
    w = wl.weight(m, n, 0.02, 31)
    x = torch.randn(2 * n, n, device=dev(), generator=torch.Generator(device=dev()).manual_seed(7))
    H32 = (x.T @ x / (2 * n)).cpu().numpy()
    U, dead, _ = gpu_factor(H32)
    U32, h32, s_g = U.astype(np.float32), np.ascontiguousarray(np.diag(H32)), 4e-5
    codes, packed = gpu_gptq(w, U32, h32, s_g, 128, 4, 4)
    for r0, r1 in ((0, 128), (m // 2 - 57, m // 2 + 40), (m - 200, m)):
        c, p = gpu_gptq(w[r0:r1].contiguous(), U32, h32, s_g, 128, 4, 4)
        assert np.array_equal(c, codes[r0:r1]) and np.array_equal(p, packed[r0:r1])


@pytest.mark.parametrize("m,n,block", [
    (300, 1024, 512),   # the update after a panel of one block
    (200, 1536, 768),   # after a block wider than a panel
    (300, 512, 128),    # inside a panel
    (300, 480, 32),     # inside a panel, many blocks
])
def test_gptq_propagation_keeps_fp32_accuracy(m, n, block):
    """What the propagated errors add to the weights right of them, against the same sums at 64 bits.
    The call leaves in its workspace the running weights as each panel found them and, split, the last
    panel's errors E, from which the running weights inside it follow.  The tensor cores' sums lose up
    to about a unit in the last place per 16 of K, at most 2.9e-6 over 768; measured 2.4e-7 to 1.03e-6,
    bounded by 1.6e-6.  U cut to two bf16 parts in the sums here (2.4e-6) breaks that, so the loss of
    a product would show."""
    w = wl.weight(m, n, 0.02, 41, dev())
    g = torch.Generator(device=dev()).manual_seed(n)
    U = torch.triu(torch.randn(n, n, generator=g, device=dev()), 1)
    if n <= 512:
        U *= 0.1  # the errors feed each other inside the panel
    U.diagonal().copy_(1.0 + torch.rand(n, generator=g, device=dev()))
    h, sg = torch.ones(n, device=dev()), torch.tensor([4e-5], device=dev())
    codes = torch.empty(m, n // 16, dtype=torch.uint8, device=dev())
    packed = torch.empty(m, n // 2, dtype=torch.uint8, device=dev())
    ws = torch.empty(hs.hscale_gptq_workspace_bytes(m, n, block), dtype=torch.uint8, device=dev())
    hs.hscale_gptq_hscale(w, U, h, sg, None, block, 4, 4, codes, packed, ws)
    grid = torch.tensor([0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0], dtype=torch.float64, device=dev())
    nib = torch.stack([packed & 15, packed >> 4], -1).view(m, n).long()
    scale = (codes.view(torch.float8_e4m3fn).double() * sg.double()).repeat_interleave(16, 1)
    what = torch.where((nib & 8) != 0, -1.0, 1.0).double() * grid[nib & 7] * scale
    d = torch.diagonal(U).double()
    if n > 512:
        E = (w.double() - what)[:, :block] / d[:block]          # the first block's weights are w
        got = ws[:4 * m * n].view(torch.float32).view(m, n)[:, block:].double()
        cols = [(block, n)]
    else:
        at = (4 * m * n + 255) // 256 * 256
        E = ws[at:at + 6 * m * n].view(torch.bfloat16).view(m, 3, n).double().sum(1)
        got = (E * d + what)[:, block:]
        cols = [(c, c + block) for c in range(block, n, block)]

    def distance(V):
        added = torch.cat([-(E[:, :a] @ V[:a, a:b]) if n <= 512 else -(E @ V[:block, a:b]) for a, b in cols], 1)
        return float((got - w[:, block:].double() - added).norm() / added.norm())

    hi = U.to(torch.bfloat16).float()
    two_parts = hi.double() + (U - hi).to(torch.bfloat16).double()
    rel, planted = distance(U.double()), distance(two_parts)
    print(f"[parity] gptq propagation {m} x {n}, block {block}: {rel:.2e} from 64 bits (U in two parts {planted:.2e})")
    assert rel <= 1.6e-6 < planted
    assert hs.hscale_device_error_flags() == 0


def test_gptq_zero_groups_keep_the_initial_code():
    """Groups that are all zero (dead channels) score zero under every code: the tie rule keeps
    the initial code, 1, and the nibbles are zero."""
    m, n, block = 40, 256, 64
    w, x, H, U32, h32, dead = layer_inputs(m, n, 77)
    dead = np.zeros(n, dtype=bool)
    dead[96:128] = True
    wb = bits(w)
    s_g, _ = oracle.global_scale(wb)
    Ud = np.diag(np.diag(U32)).astype(np.float32)  # nothing is propagated into the dead channels
    codes, packed = gpu_gptq(w, Ud, h32, s_g, block, 4, 4, dead=dead)
    assert np.all(codes[:, 6:8] == 1) and np.all(packed[:, 48:64] == 0)


def test_full_size_gptq_q_proj_slice():
    """A 1024 x 4096 slice of the q_proj layer at full width with the full pipeline on the
    GPU (H on the tensor cores, the factor, block loop of 128 columns, k = 4) against
    the oracle fed the GPU-independent inputs; output errors of GPTQ + H-Scale, H-Scale and
    RTN are reported."""
    W = wl.WORKLOADS["llama8b-q_proj"]
    n = 4096
    w = wl.weight(4096, n, W.sigma_w, W.seed)[:1024].contiguous()
    wb = bits(w)
    a = wl.channel_magnitudes(n, W.sigma_a, W.outlier_channels, W.outlier_channel_mult, W.seed)
    x = wl.activation_chunk(1024, a, W.seed, 0)
    H = oracle_H(x, n)
    H32 = H.astype(np.float32)
    s_g, _ = oracle.global_scale(wb)
    # GPU: H, factor, block loop
    Hg = torch.zeros(n, n, dtype=torch.float32, device=dev())
    hs.hscale_hessian_full_accumulate(x.to(dev()), Hg)
    torch.cuda.synchronize()
    scale = np.sqrt(np.outer(np.diag(H), np.diag(H)))
    assert np.all(np.triu(np.abs(Hg.cpu().double().numpy() - H)) <= 1e-5 * scale + 1e-30)
    # the factor of the GPU's own H (upper triangle only) equals the factor of the oracle's
    Ug, _, info_g = gpu_factor(Hg.cpu().numpy())
    assert np.all(info_g == 0)
    U, dead, info = gpu_factor(H32)
    assert np.all(info == 0)
    Uref, dref = oracle.gptq_factor(H32.astype(np.float64))
    assert np.linalg.norm(U - Uref) / np.linalg.norm(Uref) <= 1e-3
    assert np.linalg.norm(Ug - Uref) / np.linalg.norm(Uref) <= 1e-3
    h32 = np.diag(H32).copy()
    U32 = Uref.astype(np.float32)
    codes, packed = gpu_gptq(w, U32, h32, s_g, 128, 4, 4, dead=dref)
    ref = oracle.gptq_hscale(wb, U32.astype(np.float64), h32, s_g, 128, 4, 4, dead=dref)
    xe = x[:512].float().double().numpy()
    err = {}
    for name, c, p in (("gpu", codes, packed), ("oracle", ref["codes"], ref["packed"])):
        err[name] = oracle.output_error(xe, oracle.dequant_residual(wb, s_g, c, p))
    hsr = oracle.refine(wb, h32, s_g, None, 4, 4)
    err["hscale"] = oracle.output_error(xe, oracle.dequant_residual(wb, s_g, hsr["codes"], hsr["packed"]))
    rc = oracle.rtn_codes(wb, s_g)
    err["rtn"] = oracle.output_error(xe, oracle.dequant_residual(wb, s_g, rc, oracle.pack(wb, s_g, rc)))
    agree = float(np.mean(codes == ref["codes"]))
    print(f"[parity] gptq q_proj 1024x4096: codes equal {agree:.2%}; output error gpu {err['gpu']:.5e} "
          f"oracle {err['oracle']:.5e} hscale {err['hscale']:.5e} rtn {err['rtn']:.5e}")
    assert agree >= 0.98
    assert abs(err["gpu"] - err["oracle"]) <= 0.01 * err["oracle"]


def test_gptq_is_deterministic_and_capturable():
    """The block loop, whose kernels are scheduled while the one before them runs, gives the same
    bytes on every run, and the same bytes again when the call is captured into a CUDA graph and
    replayed."""
    m, n, block = 256, 1024, 64
    w, x, H, U32, h32, dead = layer_inputs(m, n, 123, tokens=1024)
    wb = bits(w)
    s_g, _ = oracle.global_scale(wb)
    runs = [gpu_gptq(w, U32, h32, s_g, block, 4, 4) for _ in range(3)]
    for c, p in runs[1:]:
        assert np.array_equal(c, runs[0][0]) and np.array_equal(p, runs[0][1])
    wd = w.to(dev())
    Ud = torch.from_numpy(np.ascontiguousarray(U32)).to(dev())
    hd = torch.from_numpy(h32).to(dev())
    sg = torch.tensor([s_g], dtype=torch.float32, device=dev())
    codes = torch.zeros(m, n // 16, dtype=torch.uint8, device=dev())
    packed = torch.zeros(m, n // 2, dtype=torch.uint8, device=dev())
    ws = torch.empty(hs.hscale_gptq_workspace_bytes(m, n, block), dtype=torch.uint8, device=dev())
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        hs.hscale_gptq_hscale(wd, Ud, hd, sg, None, block, 4, 4, codes, packed, ws)
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(codes.cpu().numpy(), runs[0][0])
    assert np.array_equal(packed.cpu().numpy(), runs[0][1])
    ref = oracle.gptq_hscale(wb, U32.astype(np.float64), h32, s_g, block, 4, 4, dead=dead)
    assert float(np.mean(runs[0][0] == ref["codes"])) >= 0.98


def test_factor_is_deterministic_and_capturable():
    """The factor gives the same bits on every run and when captured into a CUDA graph and
    replayed (the bench times it that way)."""
    n = 1000
    g = np.random.default_rng(31)
    A = g.standard_normal((n, n)) / np.sqrt(n)
    H32 = (A @ A.T + 0.1 * np.eye(n)).astype(np.float32)
    outs = [gpu_factor(H32) for _ in range(2)]
    assert np.array_equal(outs[0][0], outs[1][0]) and np.all(outs[0][2] == 0)
    Hd = torch.from_numpy(H32).to(dev())
    U = torch.zeros(n, n, dtype=torch.float32, device=dev())
    dead = torch.empty(n, dtype=torch.uint8, device=dev())
    info = torch.zeros(3, dtype=torch.int32, device=dev())
    ws = torch.empty(hs.hscale_gptq_factor_workspace_bytes(n), dtype=torch.uint8, device=dev())
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    gr = torch.cuda.CUDAGraph()
    with torch.cuda.graph(gr, stream=s):
        hs.hscale_gptq_factor(Hd, 0.01, U, dead, info, ws)
    gr.replay()
    torch.cuda.synchronize()
    assert np.array_equal(U.cpu().numpy(), outs[0][0]) and int(info.abs().sum()) == 0
