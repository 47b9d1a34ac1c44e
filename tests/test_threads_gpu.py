"""Threads with contexts of their own on one GPU: launches of the same kernels that differ in shared memory."""
import threading

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("variant,ks", [(4, (9, 16)), (0, (9, 16)), (5, (2, 16))])
def test_two_contexts_search_side_by_side(kb, variant, ks):
    st = synth.small_stack(77, 4, 24, 70, K=5, n_angles=4, n_speeds=2, s_hi=20.0, n_sources=1, flux=40.0)
    sci, var = torch.from_numpy(st.sci).to(DEV), torch.from_numpy(st.var).to(DEV)
    failed, records = [], [[] for _ in ks]
    start = threading.Barrier(len(ks))

    def work(i):
        try:
            ctx, stream = kb.Context(0), torch.cuda.Stream()
            ctx.set_search_variant(variant)
            s = kb.Stack(ctx, 4, 24, 70, "f32")
            s.make_psi_phi(sci, var, None, st.psf, stream=stream)
            job = kb.Job(ctx, 24, 70, 4, st.vx.size, ks[i])
            start.wait()
            for n in range(600):
                job.search(s, st.times, st.vx, st.vy, ks[i], stream=stream)
                if n % 200 == 0:
                    records[i].append(job.results(stream=stream).tobytes())
            stream.synchronize()
            job.free()
            s.free()
            ctx.close()
        except Exception as e:   # reported by the main thread
            failed.append((ks[i], repr(e)))

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(ks))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
    assert all(len(r) == 3 and len(set(r)) == 1 for r in records)
