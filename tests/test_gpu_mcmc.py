"""GPU parity of MCMC relocation (ubs_mcmc_relocate) against the reference:
the drawn sources bit for bit, copied parameters bit for bit, the cloned
opacities within float32 rounding, and the reset moments."""
import numpy as np
import pytest
import torch

from oracle import mcmc64 as M
from paper_2510_03312_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_03312_gb300 import build as B
    B.build()
    return torch.device("cuda", 0)


def _case(P, seed, dead_frac):
    rng = np.random.default_rng(seed)
    sc = S.make_scene(seed, 6, P)
    act = sc.params.copy()
    orow = sc.offsets()["opacity"][0]
    o = act[orow]
    dead = rng.random(P) < dead_frac
    o[dead] = rng.uniform(0.0, 0.005, dead.sum()).astype(np.float32)
    raw = act.copy()
    raw[orow] = np.log(o / (1 - o))
    m = rng.standard_normal(act.shape).astype(np.float32)
    v = rng.random(act.shape).astype(np.float32)
    rand = rng.integers(0, 2 ** 63, size=P, dtype=np.uint64) * np.uint64(2) + rng.integers(0, 2, size=P,
                                                                                            dtype=np.uint64)
    return act, raw, m, v, rand, orow


@pytest.mark.parametrize("P,seed,dead_frac", [(3000, 1, 0.1), (5000, 2, 0.6), (1024, 3, 0.05), (1, 4, 0.0),
                                              (200_000, 5, 0.02), (777, 6, 1.0)])
def test_relocation_matches_reference(dev, P, seed, dead_frac):
    from paper_2510_03312_gb300 import ubs as U
    import ctypes
    act, raw, m, v, rand, orow = _case(P, seed, dead_frac)
    K = act.shape[0]
    t = {k: torch.tensor(a, device=dev).contiguous() for k, a in dict(act=act, raw=raw, m=m, v=v).items()}
    rnd = torch.tensor(rand.view(np.int64), device=dev)
    src = torch.empty(P, dtype=torch.int32, device=dev)
    nrel = torch.zeros(1, dtype=torch.int64, device=dev)
    n = U.ubs_mcmc_workspace_size(P)
    ws = torch.empty(n + 256, dtype=torch.uint8, device=dev)
    wp = (ws.data_ptr() + 255) // 256 * 256
    st = U.ubs_mcmc_relocate(K, P, orow, 0.005, t["act"].data_ptr(), t["raw"].data_ptr(), t["m"].data_ptr(),
                             t["v"].data_ptr(), rnd.data_ptr(), src.data_ptr(), nrel.data_ptr(), wp, n,
                             ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == U.UBS_OK
    a_r, r_r, m_r, v_r, src_r = M.relocate(act, raw, m, v, orow, rand)
    s_g = src.cpu().numpy()
    assert np.array_equal(s_g, src_r)
    assert int(nrel.item()) == int((src_r >= 0).sum())
    ag, rg = t["act"].cpu().numpy(), t["raw"].cpu().numpy()
    other = [k for k in range(K) if k != orow]
    assert np.array_equal(ag[other], a_r[other].astype(np.float32))
    assert np.array_equal(rg[other], r_r[other].astype(np.float32))
    np.testing.assert_allclose(ag[orow], a_r[orow], rtol=2e-6, atol=1e-9)
    touched = (src_r >= 0) | (np.bincount(src_r[src_r >= 0], minlength=P) > 0)
    np.testing.assert_allclose(rg[orow][touched], r_r[orow][touched], rtol=2e-5, atol=2e-5)
    assert np.array_equal(rg[orow][~touched], raw[orow][~touched])
    assert np.array_equal(t["m"].cpu().numpy(), m_r.astype(np.float32))
    assert np.array_equal(t["v"].cpu().numpy(), v_r.astype(np.float32))


@pytest.mark.parametrize("P,dead_frac", [(32, 0.5), (33, 0.5), (32 * 1024, 0.01), (32 * 1024 + 1, 0.3),
                                         (1024 * 1024 + 1, 0.02)])
def test_draw_search_at_its_level_edges(dev, P, dead_frac):
    """The 32-way search of a draw at the edges of its levels: one chunk of 32,
    32 blocks of 1024 and one more, 1024 blocks and one more (a third level),
    with runs of zero weights; the sources against the cumulative weights by
    definition, bit for bit.  One plane, the opacity."""
    import ctypes

    from paper_2510_03312_gb300 import ubs as U
    rng = np.random.default_rng(P)
    o = rng.random(P).astype(np.float32)
    o[rng.random(P) < dead_frac] = 0.0
    o[P // 4:P // 2] = 0.0  # whole chunks and blocks without weight
    o[-1] = 1.0
    o[0] = 0.0
    rand = rng.integers(0, 2 ** 63, size=P, dtype=np.uint64) * np.uint64(2) + np.uint64(1)
    dead = o <= np.float32(0.005)
    w = np.where(dead, 0, np.floor(o.astype(np.float64) * 2 ** 24)).astype(np.uint64)
    cum = np.cumsum(w, dtype=np.uint64)
    want = np.where(dead, np.searchsorted(cum, rand % cum[-1], side="right"), -1).astype(np.int32)
    act, raw = torch.tensor(o, device=dev)[None].contiguous(), torch.zeros(1, P, device=dev)
    m, v = torch.ones(1, P, device=dev), torch.ones(1, P, device=dev)
    rnd = torch.tensor(rand.view(np.int64), device=dev)
    src = torch.empty(P, dtype=torch.int32, device=dev)
    nrel = torch.zeros(1, dtype=torch.int64, device=dev)
    n = U.ubs_mcmc_workspace_size(P)
    ws = torch.empty(n + 256, dtype=torch.uint8, device=dev)
    st = U.ubs_mcmc_relocate(1, P, 0, 0.005, act.data_ptr(), raw.data_ptr(), m.data_ptr(), v.data_ptr(),
                             rnd.data_ptr(), src.data_ptr(), nrel.data_ptr(), (ws.data_ptr() + 255) // 256 * 256, n,
                             ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == U.UBS_OK
    assert np.array_equal(src.cpu().numpy(), want)
    assert int(nrel.item()) == int(dead.sum())
    copies = np.bincount(want[dead], minlength=P)
    new = 1.0 - (1.0 - o.astype(np.float64)) ** (1.0 / (copies + 1))
    ref = np.where(dead, new[np.maximum(want, 0)], np.where(copies > 0, new, o))
    # 1 - powf(1 - o, 1 / (n + 1)): a few roundings of numbers up to 1
    np.testing.assert_allclose(act[0].cpu().numpy(), ref, rtol=2e-6, atol=5e-7)
    moved = dead | (copies > 0)
    assert np.array_equal(m[0].cpu().numpy(), np.where(moved, 0.0, 1.0).astype(np.float32))
    assert np.array_equal(v[0].cpu().numpy(), np.where(moved, 0.0, 1.0).astype(np.float32))


@pytest.mark.parametrize("P,dead_frac", [(31, 0.5), (63, 0.5), (64, 0.5), (65, 0.5), (1023, 0.3), (1024, 0.95),
                                         (1025, 0.95), (19_455, 0.2), (19_457, 0.95), (311_295, 0.95),
                                         (311_297, 0.05), (1024 * 1024, 0.02), (3 * 1024 * 1024 + 1, 0.01)])
def test_draw_at_chunk_and_block_edges(dev, P, dead_frac):
    """The draw at the edges of its chunks of 64 and blocks of 1024
    primitives, of the slots a CTA takes (64 to 1024 by the scene's size) and
    of the staged block offsets (every one up to 1M primitives, then every
    second and fourth), with few and with nearly all slots dead."""
    test_draw_search_at_its_level_edges(dev, P, dead_frac)


@pytest.mark.parametrize("P", [64, 1024, 4096, 1500 * 1024])
@pytest.mark.parametrize("live", ["last_of_four", "second_half", "one_per_chunk", "one_per_block", "last_block"])
def test_draw_among_few_live_primitives(dev, P, live):
    """Weights in one place of each group the draw searches: the last of a
    lane's four, the second half of a chunk, one primitive a chunk or a block,
    and the last block only (whole staged steps without weight before it): the
    sources against the cumulative weights by definition, bit for bit."""
    import ctypes

    from paper_2510_03312_gb300 import ubs as U
    rng = np.random.default_rng(P)
    i = np.arange(P)
    on = {"last_of_four": i % 4 == 3, "second_half": i % 64 >= 32, "one_per_chunk": i % 64 == (i // 64 * 7) % 64,
          "one_per_block": i % 1024 == min(P, 1024) - 1, "last_block": i >= P - min(P // 2, 1024)}[live]
    o = np.where(on, rng.uniform(0.006, 1.0, P), 0.0).astype(np.float32)
    rand = rng.integers(0, 2 ** 63, size=P, dtype=np.uint64) * np.uint64(2) + np.uint64(1)
    w = np.where(on, np.floor(o.astype(np.float64) * 2 ** 24), 0).astype(np.uint64)
    cum = np.cumsum(w, dtype=np.uint64)
    rand[:2] = 0, cum[-1] - np.uint64(1)  # the first and the last unit of weight
    want = np.where(on, -1, np.searchsorted(cum, rand % cum[-1], side="right")).astype(np.int32)
    act, raw, m, v = (torch.tensor(a, device=dev)[None].contiguous() for a in (o, 0 * o, 0 * o, 0 * o))
    rnd = torch.tensor(rand.view(np.int64), device=dev)
    src = torch.empty(P, dtype=torch.int32, device=dev)
    nrel = torch.zeros(1, dtype=torch.int64, device=dev)
    n = U.ubs_mcmc_workspace_size(P)
    ws = torch.empty(n + 256, dtype=torch.uint8, device=dev)
    st = U.ubs_mcmc_relocate(1, P, 0, 0.005, act.data_ptr(), raw.data_ptr(), m.data_ptr(), v.data_ptr(),
                             rnd.data_ptr(), src.data_ptr(), nrel.data_ptr(), (ws.data_ptr() + 255) // 256 * 256, n,
                             ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == U.UBS_OK
    assert np.array_equal(src.cpu().numpy(), want)
    assert int(nrel.item()) == int((~on).sum())
