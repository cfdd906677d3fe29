"""B200-native fused dequantize + matrix-vector product over block-quantised weights.

The public calls (`matvec`, `dequant`, `quantize`, ...) live in `paper_2605_20706_b200.lw`, a thin
Python binding over the C-ABI shared library built from `csrc/`.  `synth` holds the seeded input
generators and the Llama-shaped decode-step shape lists.
"""
