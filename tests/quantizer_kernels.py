"""Which quantizer kernel a call takes: reads a JSON list of calls from standard input, prints the kernels' names as JSON.  A program of its
own, since the profiler records nothing any more once other tests have run in its process.  A call: M, K, block, a_bits, what ("codes", "operand"),
and optionally "smooth" (multipliers), "offset" (bytes of the codes from a 256-byte boundary)."""
import json
import sys

import torch
from torch.profiler import ProfilerActivity, profile

import paper_2508_03485_b200 as P


def call(c):
    M, K = c["M"], c["K"]
    X = torch.randn((M, K), device="cuda", dtype=torch.bfloat16)
    pre = torch.ones(K, device="cuda") if c.get("smooth") else None
    if c["what"] == "operand":
        tlq = P.lrq_tlq_quantize_weights(0.02 * torch.randn((32, K), device="cuda"), 4, 0, 7, [1.0], [1.0])
        layer = P.QLayer(tlq, 32, K, P.ROT_HADAMARD, c["a_bits"], c["block"], prescale=pre)
        return lambda: P.lrq_qlinear(layer, X, P.BF16)
    out = None
    if "offset" in c:
        out = (torch.empty(M * K * c["a_bits"] // 8 + c["offset"], device="cuda", dtype=torch.uint8)[c["offset"]:],
               torch.empty(M, device="cuda"), torch.empty(M, device="cuda", dtype=torch.int32))
    return lambda: P.lrq_rotate_quantize_act(X, P.ROT_HADAMARD, c["a_bits"], c["block"], prescale=pre, out=out)


names = []
for c in json.load(sys.stdin):
    f = call(c)
    f()
    found = []
    for _ in range(5):                       # a profile of one short call comes back empty now and then: it is taken again
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            f()
            torch.cuda.synchronize()
        found = [e.name for e in prof.events() if "rotq_" in e.name]
        if found:
            break
    assert len(found) == 1, (c, found)
    names.append(found[0])
print(json.dumps(names))
