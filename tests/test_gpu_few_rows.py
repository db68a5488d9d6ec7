"""Calls that take kernels of their own by their size, at the edges of their ranges: the
role-routed linear map of few rows (the row paddings 16, 32, 64, 128, 192, with and without a
split of the reduction, ragged column tiles, one kind of row or both; the lines by width) and of
very many; decode in equal shares; the single-launch scan of the compaction; prefills whose units
are shared by clusters of blocks; calls captured behind copies and memsets."""
import numpy as np
import pytest
import torch

from paper_2601_21927_gb300 import inputs, sonic
from tests import harness as H
from tests.test_gpu_compact import _check as _check_compact
from tests.test_gpu_compact import _run as _compact
from tests.test_gpu_decode import _check as _check_decode
from tests.test_gpu_decode import _check_mass, _decode
from tests.test_gpu_routed import _check, _roles, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 16, 17, 32, 33, 64, 65, 128, 129, 191, 192, 193])
def test_routed_linear_row_paddings(T):
    """Reductions of 3 steps (no split) and 16 steps (split by up to 4); 160 columns end
    inside a 128-row weight tile and inside a part."""
    for d_in, seed in ((192, 31), (1024, 32)):
        r = _run(_roles(T, T + seed), d_in, [96, 32, 32], [False, True, True], seed=seed,
                 cache_rows=2 * T + 5, x_pad=64)
        _check(r)


@pytest.mark.parametrize("role", [inputs.ROLE_CURR, inputs.ROLE_NEXUS, None])
@pytest.mark.parametrize("T,d_in,cols", [(7, 4096, [4096, 1024, 1024]), (40, 3584, [3584]),
                                         (190, 2048, [2048, 512, 512]), (130, 2112, [4640])])
def test_routed_linear_projection_widths(role, T, d_in, cols):
    roles = _roles(T, T) if role is None else np.full(T, role, np.uint8)
    r = _run(roles, d_in, cols, [False] + [True] * (len(cols) - 1), seed=41, cache_rows=T + 9)
    _check(r)


@pytest.mark.parametrize("T", [131072, 131073])
def test_routed_linear_counted_by_a_launch_of_its_own(T):
    """Both sides of the largest call whose partition counts the roles itself."""
    r = _run(_roles(T, 7), 64, [32, 32], [False, True], seed=T, cache_rows=T + 5)
    _check(r, np.r_[0:300, T // 2:T // 2 + 300, T - 300:T])


@pytest.mark.parametrize("T", [16384, 16385])
def test_routed_linear_one_kind_of_row(T):
    """Both sides of the largest call whose GEMM looks at the roles itself."""
    r = _run(np.full(T, inputs.ROLE_NEXUS, np.uint8), 64, [32, 32], [False, True], seed=T,
             cache_rows=T + 77)
    _check(r, np.r_[0:300, T // 2:T // 2 + 300, T - 300:T])


def test_routed_linear_calls_in_a_row_share_a_workspace():
    """Calls of one kind of row (whose GEMM runs beside the partition kernels) between calls of
    both kinds, back to back on one workspace."""
    T, d = 2500, 512
    W = inputs.randn((256, d), seed=1, device=H.dev())
    Wn = inputs.randn((256, d), seed=2, device=H.dev())
    X = [inputs.randn((T, d), seed=3 + k, device=H.dev()) for k in range(6)]
    roles = [np.full(T, inputs.ROLE_CURR), _roles(T, 1), np.full(T, inputs.ROLE_NEXUS), _roles(T, 2),
             np.full(T, inputs.ROLE_CURR), _roles(T, 3)]
    rt = [torch.from_numpy(r.astype(np.uint8)).to(H.dev()) for r in roles]
    Y = [torch.empty((T, 256), dtype=torch.bfloat16, device=H.dev()) for _ in X]
    ws = None
    for _ in range(20):
        for x, r, y in zip(X, rt, Y):
            y.zero_()
            ws = sonic.sonic_routed_linear(x, W, Wn, r, [(y, False)], workspace=ws)
    torch.cuda.synchronize()
    for x, r, y in zip(X, rt, Y):
        one = torch.empty_like(y)
        sonic.sonic_routed_linear(x, W, Wn, r, [(one, False)])
        torch.cuda.synchronize()
        assert torch.equal(one.view(torch.int16), y.view(torch.int16))
        want = torch.where((r == inputs.ROLE_NEXUS)[:, None], x.float() @ Wn.float().T,
                           x.float() @ W.float().T)
        # fp32 sums of 512 products of N(0, 1) values (rms 23), rounded to bf16
        assert ((y.float() - want).abs() <= 2.0 ** -8 * want.abs() + 0.1).all()


@pytest.mark.parametrize("hq,hkv,D,nl", [(32, 8, 128, 1), (28, 4, 128, 3), (4, 2, 64, 2),
                                         (3, 1, 128, 1), (16, 1, 64, 1), (30, 15, 128, 1)])
@pytest.mark.parametrize("lens", [
    [1], [16], [63, 64, 65], [128 * 19 + 31], [0, 5, 0, 700, 0], [4096, 1, 33, 31, 32, 2050],
    list(range(1, 130))], ids=lambda v: f"{len(v)}x{max(v)}")
def test_decode_equal_shares(lens, hq, hkv, D, nl):
    """Sequences shorter than a share, far longer, empty, ending next to a cut (within the
    32 keys a cut moves by), many to a block; lse and Nexus mass too."""
    r = _decode(np.array(lens, np.int32), hq, hkv, D, n_layers=nl, seed=len(lens) + hq,
                with_mass=True)
    pairs = [(nl - 1, b) for b in range(0, len(lens), 1 + len(lens) // 12)] + [(0, len(lens) - 1)]
    _check_decode(r, pairs)
    _check_mass(r, pairs)
    assert not r["O"].isnan().any()


def test_calls_captured_after_copies_and_memsets():
    """A graph whose calls follow a copy and a memset (no kernel before them): replays equal
    the eager calls bit for bit."""
    lens, starts = H.i32([700, 45]), H.i32([0, 700])
    K = inputs.randn((1, 745, 8, 128), seed=1, device=H.dev())
    V = inputs.randn((1, 745, 8, 128), seed=2, device=H.dev())
    q = inputs.randn((1, 2, 32, 128), seed=3, device=H.dev())
    W = inputs.randn((256, 4096), seed=4, device=H.dev())
    role = torch.full((2,), inputs.ROLE_CURR, dtype=torch.uint8, device=H.dev())
    qc, O = torch.empty_like(q), torch.empty_like(q)
    Y = torch.empty((2, 256), dtype=torch.bfloat16, device=H.dev())
    z = torch.empty(1 << 20, device=H.dev())

    def step(ws):
        z.zero_()
        qc.copy_(q)
        w0 = sonic.sonic_attn_decode(qc, K, V, lens, O, kv_start=starts, max_len=700,
                                     workspace=ws[0])
        z.zero_()
        return w0, sonic.sonic_routed_linear(O.view(2, 4096), W, W, role, [(Y, False)],
                                             workspace=ws[1])

    ws = step((None, None))
    torch.cuda.synchronize()
    want = O.clone(), Y.clone()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        step(ws)
    for _ in range(3):
        O.fill_(float("nan"))
        Y.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(O.view(torch.int16), want[0].view(torch.int16))
        assert torch.equal(Y.view(torch.int16), want[1].view(torch.int16))


@pytest.mark.parametrize("n_seqs,rows,total", [(1, 524288, 524288), (1, 524289, 524289),
                                               (128, 2048, 1 << 18), (128, 2049, 128 * 2049),
                                               (2, 2047, 0), (3, 2049, 0), (15, 900, 0),
                                               (17, 4100, 0), (40, 77, 0), (128, 300, 0)])
def test_compact_single_launch_scan(n_seqs, rows, total):
    """On both sides of the largest calls of the single-launch scan (524,288 rows; rows x sequences
    of 2^25), sequences at every alignment of the role bytes, pieces that end off the 16-byte
    words, empty and body-only sequences among the ragged ones, reserve rows."""
    rng = np.random.default_rng(rows)
    ds = []
    for k in range(n_seqs):
        n = total // n_seqs if total else int(rng.integers(1, rows + 1))
        segs, left = [], n
        while left > 700:
            b, x = int(rng.integers(0, 600)), int(rng.integers(0, 70))
            segs.append((b, x))
            left -= b + x
        ds.append(inputs.Dialogue(int(rng.integers(0, left + 1)) if not total else left, segs, 0))
    if n_seqs > 2 and not total:
        ds[1], ds[2] = inputs.Dialogue(0, [], 0), inputs.Dialogue(0, [(333, 0)], 0)
    batch = inputs.Batch(ds)
    assert not total or batch.total == total
    K = inputs.randn((1, batch.total, 1, 8), seed=rows, device=H.dev())
    V = inputs.randn((1, batch.total, 1, 8), seed=rows + 1, device=H.dev())
    reserve = rng.integers(0, 5, batch.B)
    _check_compact(batch, K, V, _compact(batch, K, V, reserve=reserve), reserve=reserve)


@pytest.mark.parametrize("mode", [sonic.NEXUS_FULL, sonic.NEXUS_CAUSAL_SEGMENTS])
@pytest.mark.parametrize("hq,hkv,D", [(8, 2, 128), (6, 2, 128), (7, 1, 64), (4, 1, 64)])
@pytest.mark.parametrize("q", [1, 30, 65, 128, 129, 257, 400])
def test_prefill_split_units(q, hq, hkv, D, mode):
    """One or two sequences of few query rows over 5 to 20 key tiles: paired, unpaired and
    packed units shared by clusters of 2 to 8 blocks, among them blocks without a key
    tile (a short sequence beside a long one), rows that see keys of some blocks only,
    with and without the optional outputs."""
    batch = inputs.Batch([inputs.Dialogue(100, [(130, 20), (260, 0), (0, 33), (400, 60)], q + 900),
                          inputs.Dialogue(0, [(5, 3), (60, 9)], q)])
    rows = np.unique(np.r_[0, q // 2, q - 1])
    for q_len in ([q, q], [min(q + 600, 1000), 0]):
        res = H.run_prefill(batch, hq, hkv, D, q_len=q_len, seed=q + hq, nexus_vis=mode,
                            with_mass=True)
        plain = H.run_prefill(batch, hq, hkv, D, q_len=q_len, nexus_vis=mode, with_lse=False,
                              K=res["K"], V=res["V"], Q=res["Q"])
        assert torch.equal(plain["O"].view(torch.int16), res["O"].view(torch.int16))
        assert torch.isfinite(res["O"].float()).all()
        for b in range(2):
            at = rows[rows < q_len[b]]
            if not len(at):
                continue
            O, lse, got, got_lse = H.oracle_prefill_rows(batch, res, b, at, nexus_vis=mode)
            H.check_close(got, O, f"seq {b}")
            np.testing.assert_allclose(got_lse, lse, rtol=0, atol=2e-3)
            want, mass = H.oracle_mass_rows(batch, res, b, at, nexus_vis=mode)
            np.testing.assert_allclose(mass, want, rtol=0, atol=2e-3)


@pytest.mark.parametrize("hq,hkv,D,n", [(2, 1, 64, 2048), (2, 1, 128, 1024), (8, 2, 128, 2048),
                                        (8, 2, 128, 1024), (3, 1, 64, 1500)])
def test_prefill_split_blocks_without_a_key_tile(hq, hkv, D, n):
    """Every row of one sequence, layer by layer: the first query blocks list fewer key tiles than
    their cluster has blocks (a block without one copies its Q for nothing, and its part of the
    rows goes over that copy).  All rows against a call over so many layers that no unit is split,
    20 times over with Q out of L2, bit for bit the same each time."""
    batch = inputs.Batch([inputs.Dialogue(400, [(200, 20), (0, 0), (300, 9)], n - 929)])
    nl = 12 * 8 // hq + 8
    res = H.run_prefill(batch, hq, hkv, D, seed=n + hq, n_layers=nl, with_mass=True)
    role, seg, k_start, k_len = H.meta(batch)
    flush = torch.empty(1 << 28, dtype=torch.uint8, device=H.dev())
    first, ws = {}, None
    for i in range(20):
        l = i % 2 * (nl - 1)
        O = torch.full_like(res["O"][:1], float("nan"))
        lse, mass = torch.full_like(res["lse"][:1], 7.0), torch.full_like(res["mass"][:1], 7.0)
        status = torch.zeros(1, dtype=torch.int32, device=H.dev())
        flush.fill_(i)
        ws = sonic.sonic_attn_prefill(
            res["Q"][l:l + 1], res["K"][l:l + 1], res["V"][l:l + 1], seg, role, O, k_start=k_start,
            k_len=k_len, q_start=k_start, q_len=k_len, max_q_len=n, max_k_len=n, lse=lse,
            nexus_mass=mass, status=status, workspace=ws)
        torch.cuda.synchronize()
        assert sonic.read_status(status) == 0
        got = (O.view(torch.int16), lse, mass)
        if l not in first:
            first[l] = got
            H.check_close(H.f64(O[0]), H.f64(res["O"][l]), f"layer {l}")
            np.testing.assert_allclose(H.f64(lse[0]), H.f64(res["lse"][l]), rtol=0, atol=2e-3)
            np.testing.assert_allclose(H.f64(mass[0]), H.f64(res["mass"][l]), rtol=0, atol=2e-3)
        assert all(torch.equal(a, b) for a, b in zip(first[l], got))


@pytest.mark.parametrize("T", [7, 150, 300, 2500])
@pytest.mark.parametrize("role", [inputs.ROLE_CURR, None])
def test_routed_linear_after_a_timeout(T, role):
    """A status word that says a wait ran out: no block starts work (whatever the block's warps do,
    they decide it from one read of the word), nothing is written; the next call is whole."""
    roles = _roles(T, T) if role is None else np.full(T, role, np.uint8)
    X = inputs.randn((T, 512), seed=1, device=H.dev())
    W = inputs.randn((320, 512), seed=2, device=H.dev())
    rt = torch.from_numpy(roles).to(H.dev())
    Y = torch.full((T, 320), float("nan"), dtype=torch.bfloat16, device=H.dev())
    status = torch.full((1,), 5, dtype=torch.int32, device=H.dev())  # SONIC_ERR_DEVICE_TIMEOUT
    ws = sonic.sonic_routed_linear(X, W, W, rt, [(Y, False)], status=status)
    torch.cuda.synchronize()
    assert sonic.read_status(status) == 5 and Y.isnan().all()
    status.zero_()
    sonic.sonic_routed_linear(X, W, W, rt, [(Y, False)], status=status, workspace=ws)
    torch.cuda.synchronize()
    assert sonic.read_status(status) == 0
    want = X.float() @ W.float().T
    # fp32 sums of 512 products of N(0, 1) values (rms 23), rounded to bf16
    assert ((Y.float() - want).abs() <= 2.0 ** -8 * want.abs() + 0.1).all()


@pytest.mark.parametrize("T", [1, 16, 192, 193, 700])
def test_routed_linear_refuses_a_misaligned_workspace(T):
    """Refused whatever the number of rows, also where the call has no use for the workspace."""
    X = inputs.randn((T, 128), seed=1, device=H.dev())
    W = inputs.randn((64, 128), seed=2, device=H.dev())
    role = torch.full((T,), inputs.ROLE_CURR, dtype=torch.uint8, device=H.dev())
    Y = torch.full((T, 64), float("nan"), dtype=torch.bfloat16, device=H.dev())
    ws = sonic.sonic_routed_linear(X, W, W, role, [(Y, False)])
    Y.fill_(float("nan"))
    buf = torch.empty(ws.numel() + 16, dtype=torch.uint8, device=H.dev())
    assert buf.data_ptr() % 16 == 0
    for offset in (1, 8):
        with pytest.raises(sonic.SonicError) as e:
            sonic.sonic_routed_linear(X, W, W, role, [(Y, False)], workspace=buf[offset:])
        assert e.value.code == 1
    torch.cuda.synchronize()
    assert Y.isnan().all()


@pytest.mark.parametrize("tiles,T", [(76, 192), (76, 193), (77, 128), (77, 129), (152, 128),
                                     (152, 129), (153, 16), (153, 17)])
def test_routed_linear_widths_at_the_lines(tiles, T):
    """Both sides of the largest call of few rows, where the 128-row weight tiles take clusters, one
    CTA each, or more than one wave (152 SMs)."""
    d_out = tiles * 128 - 96
    r = _run(_roles(T, T), 128, [d_out - 64, 64], [False, True], seed=tiles, cache_rows=T + 3)
    _check(r)
