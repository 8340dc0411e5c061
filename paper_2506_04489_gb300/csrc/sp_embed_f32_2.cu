// FP32 (and mixed) passes of sp_embed.cuh, length group 2, compiled apart to keep translation units small.
#include "sp_embed.cuh"

SP_F_GROUP2(SP_EMBED_FLOAT, )
