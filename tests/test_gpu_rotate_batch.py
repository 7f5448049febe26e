"""Several tokens per accumulator in the rotate kernel (sq_rotate_quant_tc.cu) give the bits of one token at a time."""
import numpy as np
import pytest

from gpu_util import Guarded, dev, torch_mod
from oracle import singlequant_oracle as ora

pytestmark = pytest.mark.gpu


# Four tokens side by side and two, full and ragged lane ranges, both numbers of columns.
@pytest.mark.parametrize("n1,n2", [(2, 64), (16, 64), (31, 64), (32, 64), (33, 64), (48, 64), (64, 64), (33, 128), (64, 128), (2, 128),
                                   (24, 128), (32, 128)])
@pytest.mark.parametrize("M", [17, 301])
def test_a_batch_has_the_bits_of_its_tokens(n1, n2, M):
    """Rows up to 16 are rotated one to an accumulator; the same rows within a larger batch share one, and an infinity among
    them stays in its own row."""
    from paper_2511_22316_b200 import binding as sq
    rng = np.random.default_rng(n1 * 131 + n2 + M)
    K = n1 * n2
    X = rng.standard_normal((M, K)).astype(np.float16)
    X[:, rng.choice(K, 4, replace=False)] *= 50
    bad = 5
    R1, R2 = ora.build_rotation(X[:8].astype(np.float32), n1, n2, seed=1)
    X[bad, K // 2] = np.inf
    rot = sq.sq_rotation_from_factors(R1, R2)
    dX = dev(X)

    def run(x, rows):
        q, s, z = Guarded(rows * K // 2), Guarded(rows * 2), Guarded(rows * K * 2)
        sq.sq_rotate_quant_act(rot, x, rows, q, s)
        sq.sq_rotate_act_f16(rot, x, rows, z)
        torch_mod().cuda.synchronize()
        assert sq.sq_last_device_status() == sq.SQ_OK
        for g in (q, s, z):
            g.check()
        return q.numpy(np.uint8, (rows, K // 2)), s.numpy(np.uint16, (rows,)), z.numpy(np.uint16, (rows, K))

    whole = run(dX, M)
    fine = np.arange(M) != bad
    for r0 in range(0, M, 16):
        rows = min(16, M - r0)
        part = run(dX[r0:r0 + rows], rows)
        keep = fine[r0:r0 + rows]
        for a, b in zip(whole, part):
            assert np.array_equal(a[r0:r0 + rows][keep], b[keep])
    z = whole[2].view(np.float16)
    assert np.all(np.isfinite(z[fine])) and not np.all(np.isfinite(z[bad]))
    rot.close()


@pytest.mark.parametrize("n1,n2", [(16, 64), (48, 64), (64, 64), (24, 128), (64, 128)])
def test_an_infinity_stays_in_its_row_with_the_structured_factor(n1, n2):
    """Two or four tokens on the lanes of an accumulator (sq_rotate_quant_st.cu): the other rows have the bits that they have
    without the infinity."""
    from paper_2511_22316_b200 import binding as sq
    M, K, bad = 37, n1 * n2, 5
    X = np.random.default_rng(n1 + n2).standard_normal((M, K)).astype(np.float16)
    rot = sq.sq_build_rotation(X[:8].astype(np.float32), n1, n2, flags=sq.SQ_ROT_DEFAULT | sq.SQ_ROT_APPLY_STRUCTURED, seed=1)
    assert rot.structured
    out = []
    for value in (X[bad, K // 2], np.inf):
        X[bad, K // 2] = value
        q, s = Guarded(M * K // 2), Guarded(M * 2)
        sq.sq_rotate_quant_act(rot, dev(X), M, q, s)
        torch_mod().cuda.synchronize()
        assert sq.sq_last_device_status() == sq.SQ_OK
        q.check(), s.check()
        out.append((np.delete(q.numpy(np.uint8, (M, K // 2)), bad, 0), np.delete(s.numpy(np.uint16, (M,)), bad)))
    assert all(np.array_equal(a, b) for a, b in zip(*out))
    rot.close()


@pytest.mark.parametrize("n1,n2,M", [(24, 128, 33), (32, 128, 64), (16, 64, 33)])
def test_the_one_launch_layer_rotates_its_batch_alike(n1, n2, M):
    """Its rotating blocks find out at run time how many tokens share an accumulator: codes, steps and outputs are those of the
    kernels one after the other, an infinity in one row or not."""
    from paper_2511_22316_b200 import binding as sq
    torch, K, N, bad = torch_mod(), n1 * n2, 256, 5
    rng = np.random.default_rng(n1 + M)
    X = rng.standard_normal((M, K)).astype(np.float16)
    rots = [sq.sq_build_rotation(X[:8].astype(np.float32), n1, n2, seed=1, flags=sq.SQ_ROT_DEFAULT | f) for f in (0, sq.SQ_ROT_FUSE_DECODE)]
    Wq, sw = dev(rng.integers(0, 256, (N, K // 2), dtype=np.uint8)), dev(np.ones(N, np.float16))
    nb = sq.sq_linear_workspace_bytes(M, K)
    X[bad, K // 2] = np.inf
    before, out = sq.sq_kernel_launch_count(), []
    for rot in rots:
        ws, y = torch.zeros(nb, dtype=torch.uint8, device="cuda"), Guarded(M * N * 2)
        sq.sq_linear(rot, dev(X), M, Wq, sw, N, K, ws, nb, y)
        torch.cuda.synchronize()
        assert sq.sq_last_device_status() == sq.SQ_OK
        y.check()
        codes = ws[:M * K // 2].cpu().numpy().reshape(M, K // 2)
        out.append([np.delete(a, bad, 0) for a in (codes, y.numpy(np.uint16, (M, N)))])
    assert sq.sq_kernel_launch_count() - before == 3
    assert all(np.array_equal(a, b) for a, b in zip(*out))
    for rot in rots:
        rot.close()
