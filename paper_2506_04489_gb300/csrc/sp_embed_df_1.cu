// double-float passes of sp_embed.cuh, length group 1, compiled apart to keep translation units small.
#include "sp_embed.cuh"

SP_F_GROUP1(SP_EMBED_DF32, )
