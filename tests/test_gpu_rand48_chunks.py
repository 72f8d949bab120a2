"""rand48 with few streams: the rounds are generated in chunks, bit for bit the
series and the states that one chain per stream gives."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,R", [(6144, 64), (6144, 333), (1, 2049), (37, 1000), (311295, 65), (400001, 3)])
def test_chunked_rounds_are_the_series(oracle_mod, S, R):
    import torch
    from paper_0709_3225_gb300 import lj
    x0 = oracle_mod.srand48_state(91 + S)
    ser = oracle_mod.rand48_series(x0, 2 * R * S)
    st = torch.empty(S, dtype=torch.int64, device="cuda")
    lj.lj_rand48_seed(st, x0)
    a = lj.lj_rand48_lrand(st, R).cpu().numpy()
    b = lj.lj_rand48_drand(st, R).cpu().numpy()
    assert np.array_equal(a, (ser[:R * S] >> np.uint64(17)).astype(np.int32))
    assert np.array_equal(b, ser[R * S:].astype(np.float64) * 2.0 ** -48)
    nxt = oracle_mod.rand48_series(int(ser[-1]), S)
    assert np.array_equal(st.cpu().numpy().view(np.uint64), nxt)


def test_chunks_of_unrelated_streams(oracle_mod):
    """The streams' states need not be one series: each runs its own chain."""
    import torch
    from paper_0709_3225_gb300 import lj
    S, R = 50, 300
    states = np.random.default_rng(3).integers(0, 1 << 48, S).astype(np.int64)
    st = torch.from_numpy(states).cuda()
    out = lj.lj_rand48_lrand(st, R).cpu().numpy().reshape(R, S)
    A, C = oracle_mod.rand48_jump(S)
    for i in (0, 17, 49):
        x = int(states[i])
        for r in range(R):
            assert out[r, i] == x >> 17
            x = (A * x + C) & ((1 << 48) - 1)
        assert int(st[i]) == x
