"""A table whose arrays fit the device but whose prepared form does not is loaded all the
same, its values converted as they are read: the same results."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

pytestmark = pytest.mark.gpu


def test_load_without_room_for_the_prepared_form(oracle):
    from paper_2609_37859_gb300 import tde
    ctx = tde.Context(0)
    nr, nt, lrho, lT = 2048, 2048, (-6.0, 2.0), (1.0, 6.0)
    le = np.add.outer(0.1 * np.linspace(0, 1, nr), np.linspace(8.0, 14.0, nt))
    tab = (nr, nt, lrho, lT, le, 0.9 * le, 0.95 * le)
    rng = np.random.default_rng(6)
    n = 2000
    rho, e = 10 ** rng.uniform(*lrho, n), 10 ** rng.uniform(8.2, 13.9, n)
    rd, ed = torch.from_numpy(rho).cuda(), torch.from_numpy(e).cuda()
    o = [torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(3)]

    def invert(mode):
        eos = tde.EOS(ctx, *tab)
        eos.invert(rd, ed, T=o[0], P=o[1], cs2=o[2], mode=mode)
        torch.cuda.synchronize()
        r = [x.cpu().numpy() for x in o]
        eos.close()
        return r

    full = invert(tde.INVERT_BISECT)   # (and every kernel is loaded)
    torch.cuda.empty_cache()
    # 28 bytes an entry for the arrays, about 88 more for the prepared form
    free = torch.cuda.mem_get_info()[0]
    room = int(nr * nt * 28 * 1.9)
    held = [torch.empty(free - room, dtype=torch.uint8, device="cuda")]
    try:
        tight = [invert(m) for m in (tde.INVERT_BISECT, tde.INVERT_BISECT_PLAIN)]
    finally:
        held.clear()
        torch.cuda.empty_cache()
    for t in tight:
        assert all(np.array_equal(a, b) for a, b in zip(full, t))
